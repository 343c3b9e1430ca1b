// Forward backprojection (echo -> image), 2D and 3D: instantiation of the
// shared kernel template and the launch set-up common to all modes.
#include "tdbp_core.cuh"

#include <algorithm>
#include <cmath>

namespace sas {
namespace core {

constexpr int MAX_WAVES = 16;    // a split image takes at most so many waves of CTAs

double series_range(sas_geometry_t h, double dmax, double ymax) {
    const double err_m = 5e-6 * h->sig.c / (2.0 * M_PI * std::max(std::fabs(h->sig.fc), h->sig.fs));
    return dmax + std::max(8.0 * ymax, std::pow(0.1 * std::pow(ymax, 5.0) / err_m, 0.25));
}

int pick_pings_per_split(long long ntiles, int P, int C, long long slots, bool uneven, double overhead,
                         double sum_cost, long long max_blocks) {
    int best = P;
    double best_cost = 0.0;
    const double per_slot = (double)ntiles / (double)slots;
    for (int s = 1; s <= P && (s == 1 || s * ntiles <= max_blocks);) {
        // not below this for s splits or more: every slot's share of the pairs and of the overheads
        if (s > 1 && per_slot * ((double)P * C + s * overhead) >= best_cost) break;
        const int pps = (P + s - 1) / s, nsplit = (P + pps - 1) / pps;
        const double waves = uneven ? per_slot * nsplit + 1.0 : std::ceil(per_slot * nsplit - 1e-9);
        const double cost = waves * ((double)pps * C + overhead) + (s > 1 ? sum_cost : 0.0);
        if (s == 1 || cost < best_cost) {
            best_cost = cost;
            best = pps;
        }
        if (pps == 1) break;
        s = (P - 1) / (pps - 1) + 1;   // the next split with fewer pings a block
        // within one wave the most splits are the best
        if (!uneven && s * ntiles < slots) s = (int)std::min<long long>(P, slots / ntiles);
    }
    return best;
}

int prepare(sas_geometry_t h, const sas_grid& g, int dim3, long long slots, Setup& S, bool need_echo, int mode) {
    int TXs, TYs, TZs;
    tile_dims(dim3, TXs, TYs, TZs);
    const double dz = dim3 ? g.dz : 0.0;
    const int nz = dim3 ? g.nz : 1;
    // largest |x - x0| over a tile bounds the differential delay (|dr| <= |d| per leg)
    const double hx = 0.5 * (TXs - 1) * std::fabs(g.dx), hy = 0.5 * (TYs - 1) * std::fabs(g.dy),
                 hz = 0.5 * (TZs - 1) * std::fabs(dz);
    const double dmax = std::sqrt(hx * hx + hy * hy + hz * hz);
    // with seabed refraction a leg's length in water metres is Lipschitz with
    // constant max(1, n), n = c / c_s (a straight segment costs at most that much)
    if (h->c_sed > 0.0 && (h->beam_tan > 0.0 || h->has_vel)) {
        set_error("the refraction model does not combine with receiver motion or a beam");
        return SAS_ERR_UNSUPPORTED;
    }
    // no pixel layer below the interface, or no step in the sound speed: every
    // leg is straight, and the straight kernels (about four times as fast, with
    // the column series) give the same image (layers as layer_z forms them)
    bool refract = h->c_sed > 0.0 && h->c_sed != h->sig.c;
    if (refract) {
        volatile double z_off = (double)(nz - 1) * dz;   // rounded by itself, as layer_z does
        refract = std::max(g.z0, g.z0 + z_off) > h->z_int;
    }
    const double n_refr = refract ? h->sig.c / h->c_sed : 1.0;
    const int U = (int)std::ceil(2.0 * std::max(1.0, n_refr) * dmax * h->sig.fs / h->sig.c) + 2;
    const int elem = (h->echo_dtype == SAS_ECHO_C32_F16 || h->echo_dtype == SAS_ECHO_C32_BF16) ? 4 : 8;
    const int align = 16 / elem;
    const int npos = 2 * U + 1;
    int seglen = 2 * U + 7 + align;
    seglen = (seglen + align - 1) / align * align;
    if (seglen > 256) {
        set_error("pixel spacing too coarse: a tile's delay span needs %d samples (max 256)", seglen);
        return SAS_ERR_UNSUPPORTED;
    }
    int npos_pad = (npos + RUN - 1) / RUN * RUN;
    // spans that fit take the fixed ring layout (see tdbp_kernel's FIXED)
    if (!refract && npos_pad <= NPOS_FIXED) npos_pad = NPOS_FIXED;
    // expansion runs of the padded positions read up to sample
    // (offset < align) + npos_pad + 6 of the slot: pad the slot past the copied segment
    const int slot_samples = std::max(seglen, npos_pad + align + 6);
    const int slot_bytes = (slot_samples * elem + 127) / 128 * 128;
    // quadratic rows for 16-bit echoes in the forward pass, else cubic rows
    const int row_bytes = (mode == MODE_FORWARD && elem == 4) ? ROW24 : ROW32;
    const int nrec = refract ? (int)NREC_REFR : (int)NREC;
    const size_t smem3 = smem_bytes(slot_bytes, npos_pad, nrec, row_bytes, 3),
                 smem2 = smem_bytes(slot_bytes, npos_pad, nrec, row_bytes, 2);
    // spans are taken up to the one whose three buffers fill the block with records of
    // eight 16-byte blocks and one set of warp sums, whatever else has been added since
    constexpr size_t LIMIT = 227 * 1024;
    const size_t added = NCW * 4 * 8 + (refract ? 0 : (size_t)NRS * PAIRS * (NREC - 32) * 4);
    if (smem3 > LIMIT + added) {
        set_error("shared memory need %zu exceeds the per-block limit", smem3);
        return SAS_ERR_UNSUPPORTED;
    }
    // two Farrow buffers instead of three where three do not fit (16-bit offset gradient,
    // 2D pixels of 5.7 to 6.05 cm at 40 kHz), or where two let a second CTA onto the SM
    // (2D complex64 pixels of 1.6 to 2.4 cm: 120 -> 101 KB)
    const int nbuf = smem3 > LIMIT || (smem3 > SMEM_TWO_CTAS && smem2 <= SMEM_TWO_CTAS) ? 2 : NBUF;
    const size_t smem = nbuf == 2 ? smem2 : smem3;
    if (smem > SMEM_TWO_CTAS) slots /= 2;    // one CTA an SM
    KParams& prm = S.prm;
    prm = KParams{};
    prm.tx = h->d_tx;
    prm.rx = h->d_rx;
    prm.txs = h->d_txs;
    prm.rxs = h->d_rxs;
    prm.k_fs_c = df_split(h->sig.fs / h->sig.c);
    prm.k_t0fs = df_split(h->sig.t0 * h->sig.fs);
    prm.k_fc_c = df_split(h->sig.fc / h->sig.c);
    prm.scale = (elem == 8) ? nullptr : h->d_scale;
    prm.coef = h->d_coef;
    prm.status = h->d_status;
    prm.x0 = g.x0; prm.y0 = g.y0; prm.z0 = g.z0;
    prm.dx = g.dx; prm.dy = g.dy; prm.dz = dz;
    prm.nx = g.nx; prm.ny = g.ny; prm.nz = nz;
    prm.tiles_x = (g.nx + TXs - 1) / TXs;
    prm.tiles_y = (g.ny + TYs - 1) / TYs;
    prm.tiles_z = (nz + TZs - 1) / TZs;
    prm.P = h->P; prm.C = h->C;
    prm.t0 = h->sig.t0; prm.fs = h->sig.fs; prm.fc = h->sig.fc; prm.inv_c = 1.0 / h->sig.c;
    prm.hs_c = (float)(2.0 * h->sig.fs / h->sig.c);
    prm.wfc_c = (float)(2.0 * M_PI * h->sig.fc / h->sig.c);
    prm.hs_c2 = make_float2(prm.hs_c, prm.hs_c);
    prm.wfc_c2 = make_float2(prm.wfc_c, prm.wfc_c);
    // largest carrier phase a pixel can take from its reference: the reference in
    // [-pi, pi) plus 2 pi fc times the differential delay, which the window bound
    // U - 2 samples limits to (U - 2) / fs
    prm.phase_direct = M_PI + 2.0 * M_PI * h->sig.fc * (U - 2) / h->sig.fs <= PHASE_DIRECT_MAX;
    prm.fs2_f = (float)(2.0 * h->sig.fs);
    prm.wfc = (float)(2.0 * M_PI * h->sig.fc);
    prm.grad_scale = (float)(-2.0 / h->sig.c);
    prm.U = U; prm.npos = npos; prm.npos_pad = npos_pad; prm.seglen = seglen; prm.seg_align = align; prm.slot_bytes = slot_bytes;
    prm.nbuf = nbuf;
    prm.rotc = h->d_rotc;
    prm.beam = h->beam_tan > 0.0;
    prm.beam_tan = (float)h->beam_tan;
    prm.beam_side = (float)h->beam_side;
    prm.cull = h->d_cull;
    prm.vel = h->has_vel ? h->d_vel : nullptr;
    prm.refract = refract;
    if (refract) {
        const double r = std::max(n_refr, 1.0 / n_refr), M = r * r - 1.0;
        prm.refr_fast_sed = n_refr < 1.0;
        prm.z_int = h->z_int;
        prm.refr_n = n_refr;
        prm.refr_nf = (float)n_refr;
        prm.refr_r2 = (float)(r * r);
        prm.refr_M = (float)M;
        prm.refr_isM = M > 0.0 ? (float)(1.0 / std::sqrt(M)) : INFINITY;
        // crossing-point tolerance: 1/2000 of a carrier wavelength
        prm.refr_tol = (float)(5e-4 * h->sig.c / h->sig.fc);
    }
    prm.hx = (float)hx;
    prm.hy = (float)hy;
    prm.hz = (float)hz;
    // column series (leg_series): the slots' offsets and its least range
    const double ystep = std::fabs(dim3 ? dz : 4.0 * g.dy), ymax = 0.5 * (PX - 1) * ystep;
    const double sgn = (dim3 ? dz : g.dy) < 0.0 ? -1.0 : 1.0;
    for (int k = 0; k < PX / 2; ++k) {
        const float y = (float)(sgn * (k + 0.5) * ystep);
        float2 &a = prm.ypos[k / 2], &b = prm.yneg[k / 2], &c = prm.ysq[k / 2];
        (k & 1 ? a.y : a.x) = y;
        (k & 1 ? b.y : b.x) = -y;
        (k & 1 ? c.y : c.x) = y * y;
    }
    // The series' paths become half samples, and those radians: rounding the two
    // factors each by itself would scale the phase (up to 500 rad over a tile) by
    // up to 7e-8, so of the FP32 values next to 2 fs/c (two ulps: 1e-5 half
    // samples over a tile) the one is taken whose product with the rounded
    // radians per half sample comes nearest to 2 pi fc/c.
    {
        const double hs = 2.0 * h->sig.fs / h->sig.c, w = 2.0 * M_PI * h->sig.fc / h->sig.c;
        float f = (float)hs;
        for (int k = 0; k < 2; ++k) f = std::nextafter(f, 0.0f);
        double best = -1.0;
        for (int k = 0; k < 5; ++k, f = std::nextafter(f, INFINITY)) {
            const float r = (float)(w / (double)f);
            const double err = std::fabs((double)f * (double)r - w);
            if (best < 0.0 || err < best) {
                best = err;
                prm.hs_s = f;
                prm.ph_hs = r;
            }
        }
    }
    prm.series_rmin = (float)series_range(h, dmax, ymax);
    prm.skip_copies = h->debug_skip_copies;
    prm.wait_ns = (unsigned long long)(h->debug_wait_ms > 0 ? h->debug_wait_ms : 4000) * 1000000ull;
    const long long ntiles = (long long)prm.tiles_x * prm.tiles_y * prm.tiles_z;
    // split the pings of each tile over several CTAs (whole pings, so that every
    // (tile, ping) belongs to exactly one CTA) where that shortens the last wave
    // of CTAs: 128 pings x 4 RX -> 256^2 at 2 cm ran 320 CTAs on 152 slots (129 us a call; 84 us
    // with 7 splits on the 304 slots of two CTAs an SM), 250 x 24 -> 1500 x 1101 in BF16 945
    // tiles on 304 (12.1 ms; 11.0 ms in splits).  Filling the pipeline and writing a
    // tile cost a CTA about 12 pairs' time; adding the parts is another launch, five pairs'
    // time (3 pings x 2 RX -> one tile: 10.0 us in one part, 11.3 us in three).  With a
    // beam the CTAs compute between none and all of their pairs, so whole waves mean
    // nothing (150 x 4 -> 400 x 300 at 3 cm, 30 degrees: 288 us by whole waves, 265 us now).
    const double sum_cost = mode == MODE_FORWARD && need_echo ? 5.0 : 0.0;
    prm.pings_per_split = slots > 0 ? pick_pings_per_split(ntiles, h->P, h->C, slots, prm.beam, 12.0, sum_cost,
                                                           (long long)MAX_WAVES * slots)
                                    : h->P;
    const int nsplit = (h->P + prm.pings_per_split - 1) / prm.pings_per_split;
    prm.nsplit = nsplit;
    if (ntiles * nsplit > 0x7fffffffLL) {
        set_error("grid too large");
        return SAS_ERR_UNSUPPORTED;
    }
    S.smem = smem;
    S.blocks = (int)(ntiles * nsplit);
    S.elem = elem;
    if (!need_echo) return SAS_OK;
    return encode_echo_map(&S.map, h->d_echo, elem, h->Ns, h->P * h->C, seglen);
}

template <typename ET, bool DIM3, int MODE>
static int launch_one(const Setup& S, cudaStream_t st) {
    const bool mv = S.prm.vel != nullptr;
    auto kern = S.prm.beam ? (mv ? tdbp_kernel<ET, DIM3, MODE, true, true> : tdbp_kernel<ET, DIM3, MODE, true, false>)
                           : (mv ? tdbp_kernel<ET, DIM3, MODE, false, true> : tdbp_kernel<ET, DIM3, MODE, false, false>);
    if (S.prm.refract)   // without a beam or motion (prepare)
        kern = tdbp_kernel<ET, DIM3, MODE, false, false, true>;
    if (!S.prm.refract && !S.prm.beam && !mv && S.prm.npos_pad == NPOS_FIXED)
        kern = tdbp_kernel<ET, DIM3, MODE, false, false, false, true>;
    SAS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S.smem));
    kern<<<S.blocks, NTHREADS, S.smem, st>>>(S.map, S.prm);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

template <int MODE>
int launch_mode(const Setup& S, int echo_dtype, int dim3, cudaStream_t st) {
    switch (echo_dtype) {
        case SAS_ECHO_C64:
            return dim3 ? launch_one<float2, true, MODE>(S, st) : launch_one<float2, false, MODE>(S, st);
        case SAS_ECHO_C32_F16:
            return dim3 ? launch_one<__half2, true, MODE>(S, st) : launch_one<__half2, false, MODE>(S, st);
        case SAS_ECHO_C32_BF16:
            return dim3 ? launch_one<__nv_bfloat162, true, MODE>(S, st)
                        : launch_one<__nv_bfloat162, false, MODE>(S, st);
        default:
            set_error("no echo uploaded");
            return SAS_ERR_STATE;
    }
}

template int launch_mode<MODE_FORWARD>(const Setup&, int, int, cudaStream_t);

// image = (accumulate ? image : 0) + the parts in a fixed order.  SLICES threads a pixel,
// each over every SLICES-th part, four loads in flight: with one thread a pixel 300 parts of a
// single tile took 20 us, one load after the other.
template <int SLICES>
__global__ void __launch_bounds__(256) sum_splits_kernel(const float2* __restrict__ parts, size_t npix, int nsplit,
                                                         int accumulate, float2* __restrict__ image) {
    constexpr int W = 256 / SLICES;
    __shared__ float2 red[SLICES][W];
    const int x = threadIdx.x % W, sl = threadIdx.x / W;
    const size_t i = blockIdx.x * (size_t)W + x;
    float2 s = make_float2(0.f, 0.f);
    if (i < npix) {
        int k = sl;
        for (; k + 3 * SLICES < nsplit; k += 4 * SLICES) {
            float2 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = parts[(k + u * SLICES) * npix + i];
#pragma unroll
            for (int u = 0; u < 4; ++u) s = fadd2(s, v[u]);
        }
        for (; k < nsplit; k += SLICES) s = fadd2(s, parts[k * npix + i]);
    }
    if (SLICES > 1) {
        red[sl][x] = s;
        __syncthreads();
        if (sl == 0)
            for (int t = 1; t < SLICES; ++t) s = fadd2(s, red[t][x]);
    }
    if (sl == 0 && i < npix) {
        if (accumulate) s = fadd2(s, image[i]);
        image[i] = s;
    }
}

void sum_splits(const float2* parts, size_t npix, int nsplit, int accumulate, float2* image, cudaStream_t st) {
    if (nsplit >= 16)
        sum_splits_kernel<8><<<(unsigned)((npix + 31) / 32), 256, 0, st>>>(parts, npix, nsplit, accumulate, image);
    else
        sum_splits_kernel<1><<<(unsigned)((npix + 255) / 256), 256, 0, st>>>(parts, npix, nsplit, accumulate, image);
}

}  // namespace core

void reserve_planes(sas_geometry_t h, cudaStream_t st) {
    using namespace core;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (h->planes.p || h->P < 2 || cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)
        return;
    // a split image's planes hold at most a tile for each of its CTAs: 70 MB
    static_assert(Tile<false>::TX * Tile<false>::TY == NCONS * PX &&
                  Tile<true>::TX * Tile<true>::TY * Tile<true>::TZ == NCONS * PX, "pixels of a tile");
    const size_t bytes = sizeof(float2) * NCONS * PX * MAX_WAVES * 2 * sm_count();
    if (cudaMalloc(&h->planes.p, bytes) == cudaSuccess) {
        h->planes.bytes = bytes;
    } else {
        h->planes.p = nullptr;
        (void)cudaGetLastError();
    }
}

int launch_forward(const ForwardArgs& a) {
    core::Setup S;
    int rc = core::prepare(a.h, a.grid, a.dim3, 2LL * sm_count(), S);
    if (rc != SAS_OK) return rc;
    S.prm.image = a.image;
    S.prm.accumulate = a.accumulate;
    if (S.prm.nsplit == 1) return core::launch_mode<core::MODE_FORWARD>(S, a.h->echo_dtype, a.dim3, a.stream);
    // several CTAs a tile: each writes its part to a plane of its own, added in a
    // fixed order (with atomic additions the image depended on the CTAs' order,
    // and it had to be cleared first); at most 16 x slots tiles' worth of planes
    const size_t npix = (size_t)a.grid.nx * a.grid.ny * S.prm.nz;
    bool own = false;
    float2* parts = nullptr;
    if (call_scratch(a.h->planes, sizeof(float2) * npix * S.prm.nsplit, false, a.stream, (void**)&parts, &own) !=
        cudaSuccess) {
        (void)cudaGetLastError();   // no memory for the planes: one CTA a tile
        rc = core::prepare(a.h, a.grid, a.dim3, 0, S);
        if (rc != SAS_OK) return rc;
        S.prm.image = a.image;
        S.prm.accumulate = a.accumulate;
        return core::launch_mode<core::MODE_FORWARD>(S, a.h->echo_dtype, a.dim3, a.stream);
    }
    S.prm.image = parts;
    S.prm.split_stride = npix;
    S.prm.accumulate = 0;
    rc = core::launch_mode<core::MODE_FORWARD>(S, a.h->echo_dtype, a.dim3, a.stream);
    if (rc == SAS_OK) {
        core::sum_splits(parts, npix, S.prm.nsplit, a.accumulate, a.image, a.stream);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "sum_splits_kernel");
    }
    if (own) cudaFreeAsync(parts, a.stream);
    return rc;
}

}  // namespace sas

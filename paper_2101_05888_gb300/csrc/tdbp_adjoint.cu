// Adjoints of the backprojection on a pixel grid:
//  * the linear adjoint B^H (image -> echo), the exact transpose of the
//    forward sum:  e_adj[i][c][floor u + k] += w_k(frac u) exp(-j 2 pi fc tau) I(x);
//  * dispatch of the offset gradient (tdbp_vjp.cu).
//
// Linear adjoint over straight 2D legs: adjoint2d_kernel below.  In 3D, with a beam,
// receiver motion or refraction, one CTA per tile (warp 0 computes the reference terms
// of 32 pairs at a time, warps 1..7 own 8 pixels each).  With the Farrow form
// w_k(f) = sum_p coef[h][k][p] g^p on the half h of the sample interval the
// per-pixel work is a scatter of g^p v (v = I(x) exp(-j 2 pi fc tau)) into
// accumulators A_p[n] in shared memory, n = floor(2u) the half-sample
// index; a transposed FIR e[floor u + k] += sum_h sum_p coef[h][k][p]
// A_p[2 floor u + h] then adds each pair's segment to the echo with global
// atomics.
#include "tdbp_core.cuh"

#include <algorithm>
#include <cmath>

namespace sas {

int launch_offset_grad(sas_geometry_t h, const sas_grid& g, const float2* grad_image, double* grad_offsets,
                       cudaStream_t st);

namespace core {

// Four consecutive fields f0 .. f0 + 3 of pair pr of a field-major record.
__device__ __forceinline__ float4 rec_block(const float* rec, int f0, int pr) {
    return make_float4(rec[f0 * PAIRS + pr], rec[(f0 + 1) * PAIRS + pr], rec[(f0 + 2) * PAIRS + pr],
                       rec[(f0 + 3) * PAIRS + pr]);
}

// REFRACT: the seabed refraction model (the forward kernel's per-leg
// crossing records and per-pixel solves, evaluated the same way).
template <bool DIM3, bool REFRACT>
__global__ void __launch_bounds__(NTHREADS, 2) adjoint_kernel(const KParams p, const float2* __restrict__ img,
                                                              float2* __restrict__ eadj, int Ns) {
    using T = Tile<DIM3>;
    constexpr int KREC = REFRACT ? NREC_REFR : NREC;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int nrow = NH * p.npos;                                   // half-sample rows per pair
    float2* A = reinterpret_cast<float2*>(smem);                    // [GROUP][nrow][NP]
    float* rec = reinterpret_cast<float*>(A + GROUP * nrow * NP);   // [KREC][PAIRS], field-major
    float* coef_s = rec + KREC * PAIRS;                             // [NH][TAPS][NP]
    int* base_s = reinterpret_cast<int*>(coef_s + NH * TAPS * NP);  // [PAIRS]
    int* rfl_s = base_s + PAIRS;                                    // [PAIRS] refraction flags

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ntiles = p.tiles_x * p.tiles_y * p.tiles_z;
    const int tile = blockIdx.x % ntiles;
    const int split = blockIdx.x / ntiles;
    const int tx0 = (tile % p.tiles_x) * T::TX;
    const int ty0 = ((tile / p.tiles_x) % p.tiles_y) * T::TY;
    const int tz0 = (tile / (p.tiles_x * p.tiles_y)) * T::TZ;
    const int ping0 = min(p.P, split * p.pings_per_split);
    const int ping1 = min(p.P, ping0 + p.pings_per_split);
    const long long q0 = (long long)ping0 * p.C, q1 = (long long)ping1 * p.C;
    const int nq = (int)(q1 - q0);
    const double cx = tx0 + 0.5 * (T::TX - 1), cy = ty0 + 0.5 * (T::TY - 1), cz = tz0 + 0.5 * (T::TZ - 1);
    const double X0 = p.x0 + cx * p.dx, Y0 = p.y0 + cy * p.dy, Z0 = p.z0 + (DIM3 ? cz * p.dz : 0.0);
    // seabed refraction: the layers below the interface and the reference depth
    double Zr = Z0;
    const unsigned bmask = REFRACT ? refr_tile_layers<DIM3>(p, tz0, Z0, Zr) : 0u;
    const float r_br = REFRACT ? (float)(Zr - p.z_int) : 0.f, r_zoff = REFRACT ? (float)(Zr - Z0) : 0.f;
    const int alen = GROUP * nrow * NP;
    const int span = p.npos + TAPS - 1;            // output samples per pair segment

    for (int t = tid; t < alen; t += NTHREADS) A[t] = make_float2(0.f, 0.f);
    if (tid < NH * TAPS * NP) coef_s[tid] = (&p.coef->c[0][0][0])[tid];

    const bool consumer = warp > 0;
    const int ct = tid - 32;
    float dxv = 0.f, dyv_c = 0.f, d2c = 0.f, r_d2h = 0.f;
    float dvar[PX], dT[PX];
    float2 G[PX];
    if (consumer) {
        int lx, ly, lz;
        T::pixel(ct, 0, lx, ly, lz);
        dxv = (float)((tx0 + lx - cx) * p.dx);
        dyv_c = (float)((ty0 + ly - cy) * p.dy);
        // the varying coordinate as the forward kernel forms it (first slot plus
        // s steps, in FP32), so that both take identical beam decisions
        const float dv0 = DIM3 ? (float)((tz0 + lz - cz) * p.dz) : dyv_c;
        const float dvstep = DIM3 ? (float)p.dz : (float)(4.0 * p.dy);
        d2c = fixed_d2<DIM3>(dxv, dyv_c);
        r_d2h = REFRACT ? fixed_d2<true>(dxv, dyv_c) : 0.f;
#pragma unroll
        for (int s = 0; s < PX; ++s) {
            T::pixel(ct, s, lx, ly, lz);
            dvar[s] = fmaf((float)s, dvstep, dv0);
            dT[s] = 0.f;
            const int ix = tx0 + lx, iy = ty0 + ly, iz = tz0 + lz;
            G[s] = (ix < p.nx && iy < p.ny && iz < p.nz) ? img[((size_t)iz * p.ny + iy) * p.nx + ix]
                                                        : make_float2(0.f, 0.f);
        }
    }
    int prev_ping = -1;
    const int nstages = (nq + PAIRS - 1) / PAIRS;
    for (int k = 0; k < nstages; ++k) {
        const long long qs = q0 + (long long)k * PAIRS;
        __syncthreads();   // previous stage's records no longer in use
        if (warp == 0 && qs + lane < q1) {
            const int i = (int)((unsigned)(qs + lane) / (unsigned)p.C);
            // the forward pass's reference terms (beam decisions agree bit for bit):
            // double-float for straight legs, FP64 with refraction
            if (REFRACT) {
                const PairGeo G = pair_geo(p, X0, Y0, Z0, qs + lane, i);
                double LT0, LR0;
                rfl_s[lane] = refr_pair_blocks(p, G, p.tx[3 * (size_t)i + 2], p.rx[3 * (size_t)(qs + lane) + 2], bmask,
                                               Zr, Z0, rec + lane, PAIRS, LT0, LR0);
                base_s[lane] = pair_record(p, G, rec + lane, PAIRS, LT0, LR0);
            } else {
                const float2 a = df_split(X0), b = df_split(Y0), c = df_split(Z0);
                const dfl X0d[3] = {dfl{a.x, a.y}, dfl{b.x, b.y}, dfl{c.x, c.y}};
                base_s[lane] = pair_record_df(p, pair_geo_df(p, X0d, (int)(qs + lane), i), rec + lane, PAIRS,
                                              p.vel ? p.vel + 3 * (size_t)i : nullptr);
            }
        }
        __syncthreads();
        float r[F_NT + 1];
#pragma unroll
        for (int f = 0; f <= F_NT; ++f) r[f] = rec[f * PAIRS + lane];
        const int npairs = (int)min((long long)PAIRS, q1 - qs);
        for (int g0 = 0; g0 < npairs; g0 += GROUP) {
            if (consumer) {
                for (int j = 0; j < GROUP && g0 + j < npairs; ++j) {
                    const int pr = g0 + j;
                    const int ping = (int)((qs + pr) / p.C);
                    if (ping != prev_ping) {
                        prev_ping = ping;
                        const float tT0 = __shfl_sync(0xffffffffu, r[F_TX], pr);
                        const float tT1 = __shfl_sync(0xffffffffu, r[F_TY], pr);
                        const float tT2 = __shfl_sync(0xffffffffu, r[F_TZ], pr);
                        const float nT2 = __shfl_sync(0xffffffffu, r[F_NT2], pr);
                        const float nT = __shfl_sync(0xffffffffu, r[F_NT], pr);
                        const float Ax = fixed_dot<DIM3>(tT0, tT1, dxv, dyv_c);
                        // seabed refraction of the transmitter leg
                        const bool trefr = REFRACT && (rfl_s[pr] & FL_T_REFR);
                        float4 tr0 = make_float4(0.f, 0.f, 0.f, 0.f), tr1 = tr0, tr2 = tr0;
                        float rhoT = 0.f, drhoT = 0.f;
                        if (REFRACT && trefr) {
                            tr0 = rec_block(rec, F_TREF, pr);
                            tr1 = rec_block(rec, F_TREF + 4, pr);
                            tr2 = rec_block(rec, F_TREF + 8, pr);
                            if (DIM3) refr_rho(tr0, Ax + r_d2h, rhoT, drhoT);
                        }
#pragma unroll
                        for (int s = 0; s < PX; ++s) {
                            const float d2 = fmaf(dvar[s], dvar[s], d2c);
                            const float a = __fadd_rn(fmaf(DIM3 ? tT2 : tT1, dvar[s], d2), Ax);
                            const float sm = nT2 + a;
                            dT[s] = a * rcp_sfu(fmaf(sm, rsqrt_sfu(sm), nT));
                            if (REFRACT && trefr) {
                                if ((bmask >> s) & 1u) {
                                    if (!DIM3) refr_rho(tr0, a, rhoT, drhoT);
                                    const float db = DIM3 ? dvar[s] - r_zoff : 0.f, b = fmaxf(r_br + db, 1e-7f);
                                    float uxi, ua;
                                    dT[s] = refr_leg_diff(p, tr0, tr1, tr2, rhoT, drhoT, b, db, r_br, uxi, ua);
                                } else {
                                    dT[s] += tr2.w;
                                }
                            }
                        }
                    }
                    const float tRx = __shfl_sync(0xffffffffu, r[F_RX], pr);
                    const float tRy = __shfl_sync(0xffffffffu, r[F_RY], pr);
                    const float tRz = __shfl_sync(0xffffffffu, r[F_RZ], pr);
                    const float nR2 = __shfl_sync(0xffffffffu, r[F_NR2], pr);
                    const float nR = __shfl_sync(0xffffffffu, r[F_NR], pr);
                    const float ufc = __shfl_sync(0xffffffffu, r[F_UF], pr);
                    const float phr = __shfl_sync(0xffffffffu, r[F_PH], pr);
                    const float Ax = fixed_dot<DIM3>(tRx, tRy, dxv, dyv_c);
                    // receiver motion: (R_R + d).v / c = Km + d_var v_var / c, as the forward
                    // kernel forms it; the beam test keeps the ping-time receiver vector
                    float Km = 0.f, vv = 0.f, bRx = tRx, bRy = tRy, bRz = tRz;
                    if (p.vel) {
                        const float* rp = rec + pr;
                        Km = DIM3 ? fmaf(rp[F_VX * PAIRS], dxv, fmaf(rp[F_VY * PAIRS], dyv_c, rp[F_RV * PAIRS]))
                                  : fmaf(rp[F_VX * PAIRS], dxv, rp[F_RV * PAIRS]);
                        vv = DIM3 ? rp[F_VZ * PAIRS] : rp[F_VY * PAIRS];
                        bRx = rp[F_BRX * PAIRS];
                        bRy = rp[F_BRY * PAIRS];
                        bRz = rp[F_BRZ * PAIRS];
                    }
                    float2* Aj = A + j * nrow * NP;
                    // seabed refraction of the receiver leg
                    const bool rrefr = REFRACT && (rfl_s[pr] & FL_R_REFR);
                    float4 rr0 = make_float4(0.f, 0.f, 0.f, 0.f), rr1 = rr0, rr2 = rr0;
                    float rhoR = 0.f, drhoR = 0.f;
                    if (REFRACT && rrefr) {
                        rr0 = rec_block(rec, F_RREF, pr);
                        rr1 = rec_block(rec, F_RREF + 4, pr);
                        rr2 = rec_block(rec, F_RREF + 8, pr);
                        if (DIM3) refr_rho(rr0, Ax + r_d2h, rhoR, drhoR);
                    }
                    float rot[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                    float tT0 = 0.f, tT1 = 0.f, tT2 = 0.f;
                    if (p.beam) {
#pragma unroll
                        for (int t = 0; t < 6; ++t) rot[t] = p.rotc[6 * (size_t)ping + t];
                        tT0 = __shfl_sync(0xffffffffu, r[F_TX], pr);
                        tT1 = __shfl_sync(0xffffffffu, r[F_TY], pr);
                        tT2 = __shfl_sync(0xffffffffu, r[F_TZ], pr);
                    }
#pragma unroll
                    for (int s = 0; s < PX; ++s) {
                        if (p.beam) {
                            // both beams must see the pixel (sensor-to-pixel vectors R + d)
                            const float dy = DIM3 ? dyv_c : dvar[s], dz = DIM3 ? dvar[s] : 0.f;
                            if (!beam_sees(p, fmaf(0.5f, tT0, dxv), fmaf(0.5f, tT1, dy), fmaf(0.5f, tT2, dz), rot) ||
                                !beam_sees(p, fmaf(0.5f, bRx, dxv), fmaf(0.5f, bRy, dy), fmaf(0.5f, bRz, dz), rot))
                                continue;
                        }
                        const float d2 = fmaf(dvar[s], dvar[s], d2c);
                        const float a = __fadd_rn(fmaf(DIM3 ? tRz : tRy, dvar[s], d2), Ax);
                        const float sm = nR2 + a;
                        const float rs = rsqrt_sfu(sm);
                        float D = fmaf(a, rcp_sfu(fmaf(sm, rs, nR)), dT[s]);
                        if (REFRACT && rrefr) {
                            if ((bmask >> s) & 1u) {
                                float rho = rhoR, drho = drhoR;
                                if (!DIM3) refr_rho(rr0, a, rho, drho);
                                const float db = DIM3 ? dvar[s] - r_zoff : 0.f, b = fmaxf(r_br + db, 1e-7f);
                                float uxi, ua;
                                D = refr_leg_diff(p, rr0, rr1, rr2, rho, drho, b, db, r_br, uxi, ua) + dT[s];
                            } else {
                                D += rr2.w;
                            }
                        }
                        if (p.vel) {
                            const float eps = fmaf(dvar[s], vv, Km) * rs;         // u_R . v / c
                            D = D * fmaf(eps, eps - 1.f, 1.f);                   // / (1 + eps)
                        }
                        const float v = fmaf(D, p.hs_c, ufc);              // 2 (u - floor u_ref) - 1/2
                        float ph = fmaf(D, p.wfc_c, phr);                  // carrier phase [rad]
                        // nearest integer of v = the half-sample index; g = frac(2u) - 1/2
                        const float t = __fadd_rn(v, FLOOR_MAGIC);
                        const float g = v - (t - FLOOR_MAGIC);
                        const unsigned pos = row_index(
                            (unsigned)(__float_as_int(t) - (__float_as_int(FLOOR_MAGIC) - NH * p.U)), (unsigned)(nrow - 1),
                            p.status);
                        if (!p.phase_direct) ph = reduce_phase(ph);
                        float sn, cs;
                        sincos_sfu(ph, sn, cs);
                        // v = G exp(-j phase)
                        float vx = fmaf(G[s].x, cs, G[s].y * sn);
                        float vy = fmaf(G[s].y, cs, -G[s].x * sn);
                        float* dst = reinterpret_cast<float*>(Aj + pos * NP);
#pragma unroll
                        for (int q = 0; q < NP; ++q) {
                            atomicAdd(dst + 2 * q, vx);
                            atomicAdd(dst + 2 * q + 1, vy);
                            vx *= g;
                            vy *= g;
                        }
                    }
                }
            }
            __syncthreads();
            // transposed FIR and flush: out[t] = sum_m sum_h sum_p coef[h][m][p] A_p[2 (t - m) + h]
            const int items = GROUP * span;
            for (int it = tid; it < items; it += NTHREADS) {
                const int j = it / span, t = it - j * span;
                const int pr = g0 + j;
                if (pr >= npairs) continue;
                const float2* Aj = A + j * nrow * NP;
                float ox = 0.f, oy = 0.f;
#pragma unroll
                for (int m = 0; m < TAPS; ++m) {
                    const int pos = t - m;
                    if (pos < 0 || pos >= p.npos) continue;
#pragma unroll
                    for (int h = 0; h < NH; ++h) {
#pragma unroll
                        for (int q = 0; q < NP; ++q) {
                            const float c = coef_s[(h * TAPS + m) * NP + q];
                            const float2 v = Aj[(NH * pos + h) * NP + q];
                            ox = fmaf(c, v.x, ox);
                            oy = fmaf(c, v.y, oy);
                        }
                    }
                }
                const long long idx = (long long)base_s[pr] + t;
                if (idx >= 0 && idx < Ns && (ox != 0.f || oy != 0.f))
                    atomicAdd(eadj + (size_t)(qs + pr) * Ns + idx, make_float2(ox, oy));
            }
            __syncthreads();
            for (int t = tid; t < alen; t += NTHREADS) A[t] = make_float2(0.f, 0.f);
        }
    }
}

// ----------------------------------------------------------------------------
// 2D, straight legs, stop-and-hop, no beam: one warp per (ping, channel) pair.
//
// The kernel above adds eight FP32 values an update with shared-memory atomics,
// which have no native form here (a compare-and-swap loop each: 14 G updates/s)
// and separates scatter, FIR and clearing by block barriers.  Here a warp owns
// its pair's accumulator rows, so that a row is updated by a plain load, add
// and store; the lanes of one instruction only have to hit different rows.
// They lie along one axis of the tile, two pixels apart, on the axis along which
// the two-way path changes faster: where neighbouring lanes' half-sample
// coordinates differ by at least one (bounded per pair from the unit vectors
// at the tile's centre and the tile's radius over the ranges) their rows are distinct.
// Pairs without that guarantee, or too near for the column series, take the
// slow form: both legs at every pixel, lanes with equal rows one after the other.
// Each lane walks lines of 32 pixels along the other axis with the column
// series of the forward pass, and keeps the sums of its current row in registers
// until the row changes.
// 128 pings x 8 RX -> 512 x 480: 17.5 ms before, 0.83 ms now (304 G updates/s);
// issue 66 % and the shared-memory pipe 60 % busy (adding every pixel to its
// row at once: 1.07 ms, that pipe 83 %).
constexpr int AT = 64;                    // tile edge [pixels]
constexpr int AIS = AT + 1;               // image row stride: lanes two rows or two columns apart, two-way conflicts
constexpr int AW = 8;                     // warps a block, one pair each
constexpr int APB = 4;                    // pairs whose records a warp forms at once
// record fields kept, and after them the low parts of 2R (x, y), |R|^2, |R| of both legs
enum { AF_RXL = F_OFF + 1, AF_RYL, AF_NR2L, AF_NRL, AF_TXL, AF_TYL, AF_NT2L, AF_NTL, AREC };
static_assert(AREC % 4 == 0, "records are read by 16-byte loads");
constexpr int ALINE = 32;                 // pixels of a line (a lane's series)
enum { AF_Y = 1, AF_SLOW = 2 };           // lanes lie along y; slow form

// One leg along a line of pixels (leg_series with its centre term in two parts).
// The lines are four times as long as a forward thread's and lie up to 45 pixels
// from the tile's centre, and an error of a pair's reference terms moves a whole
// tile coherently: with 2R, |R| and the quotient rounded to FP32 the inner
// products of the transpose were off by 2e-5 (1e-5 in the smaller tiles of the
// forward pass), so those terms carry their low parts.  (tA, tB), (tAl, tBl): 2R
// along the lanes' and the line's axis; oA, oB: the line's centre, also in two
// parts (a pixel spacing rounded to FP32 moves the tile's edge by 1e-8 m, 1e-5
// rad); (n2, n2l), (n, nl): |R|^2 and |R|.
struct LineLeg {
    float Dh, Dl, c1, c2, c3, c4;
};
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}
__device__ __forceinline__ LineLeg line_leg(float tA, float tB, float tAl, float tBl, dfl oAd, dfl oBd, float n2,
                                            float n, float n2l, float nl) {
    const float oA = oAd.hi, oB = oBd.hi;
    const float p1 = __fmul_rn(tA, oA), p2 = __fmul_rn(tB, oB), d2 = fmaf(oA, oA, oB * oB);
    float e1, e2, e3, e4;
    const float a = two_sum(two_sum(p1, p2, e1), d2, e2);            // 2R.d + |d|^2
    const float al = fmaf(tA, oA, -p1) + fmaf(tB, oB, -p2) + (e1 + e2) + fmaf(tAl, oA, tBl * oB) +
                     fmaf(tA, oAd.lo, tB * oBd.lo);
    const float sm = two_sum(n2, a, e3), sml = e3 + (n2l + al);       // |R + d|^2
    float rs = rsqrt_sfu(sm);
    rs = fmaf(0.5f * rs, fmaf(-(sm * rs), rs, 1.f), rs);
    const float hr = 0.5f * rs, r0 = sm * rs;
    const float r0l = hr * (fmaf(-r0, r0, sm) + sml);                 // |R + d| = r0 + r0l
    const float den = two_sum(r0, n, e4), rc = rcp_sfu(den);
    LineLeg L;
    L.Dh = a * rc;
    L.Dl = rc * (fmaf(-den, L.Dh, a) + fmaf(-(e4 + (r0l + nl)), L.Dh, al));
    L.c1 = fmaf(0.5f, tB, oB) * rs;
    L.c2 = hr * fmaf(-L.c1, L.c1, 1.f);
    const float q = L.c1 * rs;
    L.c3 = -(q * L.c2);
    L.c4 = fmaf(-q, L.c3, -(hr * L.c2 * L.c2));
    return L;
}

inline size_t adjoint2d_smem(int npos) {
    return sizeof(float2) * AT * AIS + sizeof(float4) * NH * TAPS +
           (size_t)AW * (sizeof(float4) * 2 * NH * npos + sizeof(float) * APB * AREC);
}

// p: with this kernel's tiles, window (U, npos) and series_rmin (lines of ALINE)
__global__ void __launch_bounds__(32 * AW, 2) adjoint2d_kernel(const KParams p, const float2* __restrict__ img,
                                                              float2* __restrict__ eadj, int Ns) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int nrow = NH * p.npos;
    float4* coef_s = reinterpret_cast<float4*>(smem);                        // [NH][TAPS] x NP
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4* rows = coef_s + NH * TAPS + (size_t)warp * 2 * nrow;             // two planes: powers 0, 1 and 2, 3
    float4* recs = coef_s + NH * TAPS + (size_t)AW * 2 * nrow;
    float* rec = reinterpret_cast<float*>(recs) + warp * APB * AREC;
    float2* im = reinterpret_cast<float2*>(reinterpret_cast<float*>(recs) + AW * APB * AREC);   // [AT][AIS]

    const int ntiles = p.tiles_x * p.tiles_y;
    const int tile = blockIdx.x % ntiles, split = blockIdx.x / ntiles;
    const int tx0 = (tile % p.tiles_x) * AT, ty0 = (tile / p.tiles_x) * AT;
    const int nx = min(AT, p.nx - tx0), ny = min(AT, p.ny - ty0);
    const long long q0 = (long long)min(p.P, split * p.pings_per_split) * p.C;
    const long long q1 = (long long)min(p.P, (split + 1) * p.pings_per_split) * p.C;
    for (int i = threadIdx.x; i < AT * AIS; i += 32 * AW) {
        const int y = i / AIS, x = i - y * AIS;
        im[i] = x < nx && y < ny ? img[(size_t)(ty0 + y) * p.nx + tx0 + x] : make_float2(0.f, 0.f);
    }
    for (int i = lane; i < 2 * nrow; i += 32) rows[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < NH * TAPS)
        coef_s[threadIdx.x] = *reinterpret_cast<const float4*>(&p.coef->c[threadIdx.x / TAPS][threadIdx.x % TAPS][0]);
    __syncthreads();
    const double X0 = p.x0 + (tx0 + 0.5 * (AT - 1)) * p.dx, Y0 = p.y0 + (ty0 + 0.5 * (AT - 1)) * p.dy;
    const float2 dx2 = df_split(p.dx), dy2 = df_split(p.dy);             // pixel spacings as double-floats
    const float2 hx2 = df_split(p.dx * (double)p.hs_s), hy2 = df_split(p.dy * (double)p.hs_s);   // in half samples
    const dfl ddx = dfl{opaque(dx2.x), opaque(dx2.y)}, ddy = dfl{opaque(dy2.x), opaque(dy2.y)};
    const dfl hdx = dfl{opaque(hx2.x), opaque(hx2.y)}, hdy = dfl{opaque(hy2.x), opaque(hy2.y)};
    const float fdx = ddx.hi, fdy = ddy.hi;
    // k pixels, k a half-integer below 64: the product in two parts
    auto times = [](float k, dfl d) {
        const float q = __fmul_rn(k, d.hi);
        return dfl{q, fmaf(k, d.hi, -q) + k * d.lo};
    };
    const float2 a_ = df_split(X0), b_ = df_split(Y0), c_ = df_split(p.z0);
    const dfl X0d[3] = {dfl{a_.x, a_.y}, dfl{b_.x, b_.y}, dfl{c_.x, c_.y}};
    const float2 magic2 = make_float2(FLOOR_MAGIC, FLOOR_MAGIC);

    // adds a[0 .. 3] to a row (lanes' rows distinct)
    auto add_row = [&](const unsigned pos, const float2* a) {
        const float4 e = rows[pos], f = rows[nrow + pos];
        const float2 s0 = fadd2(make_float2(e.x, e.y), a[0]), s1 = fadd2(make_float2(e.z, e.w), a[1]);
        const float2 s2 = fadd2(make_float2(f.x, f.y), a[2]), s3 = fadd2(make_float2(f.z, f.w), a[3]);
        rows[pos] = make_float4(s0.x, s0.y, s1.x, s1.y);
        rows[nrow + pos] = make_float4(s2.x, s2.y, s3.x, s3.y);
    };
    auto powers = [&](const float2 w, const float g, float2* a) {   // g^p w
        const float2 gg = make_float2(g, g);
        a[0] = w;
        a[1] = fmul2(w, gg);
        a[2] = fmul2(a[1], gg);
        a[3] = fmul2(a[2], gg);
    };
    // the row and weighted value of one pixel: half-sample coordinate v (t = v +
    // 1.5 2^23, g = v - rint v), phase x, image value I
    auto row_of = [&](const float t) {
        return row_index((unsigned)(__float_as_int(t) - (__float_as_int(FLOOR_MAGIC) - NH * p.U)), (unsigned)(nrow - 1),
                         p.status);
    };
    auto weighted = [&](const float x, const float2 I) {   // I exp(-j x)
        float sn, cs;
        sincos_sfu(x, sn, cs);
        return make_float2(fmaf(I.x, cs, I.y * sn), fmaf(I.y, cs, -I.x * sn));
    };

    // the warp's pairs: q0 + warp, + AW, ...
    for (long long qb = q0 + warp; qb < q1; qb += AW * APB) {
        const int cnt = (int)min((long long)APB, (q1 - qb + AW - 1) / AW);
        if (lane < cnt) {
            const int q = (int)(qb + AW * lane), i = q / p.C;
            float* rc = rec + lane * AREC;
            const PairGeoDF G = pair_geo_df(p, X0d, q, i);
            rc[F_OFF] = __int_as_float(pair_record_df(p, G, rc, 1));
#pragma unroll
            for (int leg = 0; leg < 2; ++leg) {
                // the record's fields are the double-floats' rounded values
                const dfl* g = leg ? G.T : G.R;
                const dfl n2 = df_add(df_add(df_mul(g[0], g[0]), df_mul(g[1], g[1])), df_mul(g[2], g[2]));
                const dfl n1 = df_sqrt(n2);
                float* lo = rc + (leg ? AF_TXL : AF_RXL);
                const float* hi = rc + (leg ? F_TX : F_RX);
                const float nh = rc[leg ? F_NT : F_NR];
                lo[0] = fmaf(2.f, g[0].lo, fmaf(2.f, g[0].hi, -hi[0]));
                lo[1] = fmaf(2.f, g[1].lo, fmaf(2.f, g[1].hi, -hi[1]));
                lo[2] = (n2.hi - hi[3]) + n2.lo;
                lo[3] = (n1.hi - nh) + n1.lo;
            }
            // change of the half-sample coordinate between neighbouring lanes
            // (two pixels), at least, along either axis
            const float nT = rc[F_NT], nR = rc[F_NR], dmax = sqrtf(p.hx * p.hx + p.hy * p.hy);
            const float turn = dmax / fmaxf(nT - dmax, 1e-6f) + dmax / fmaxf(nR - dmax, 1e-6f);
            const float sx = fabsf(0.5f * rc[F_TX] / nT + 0.5f * rc[F_RX] / nR);
            const float sy = fabsf(0.5f * rc[F_TY] / nT + 0.5f * rc[F_RY] / nR);
            const float vx = 2.f * fabsf(fdx) * p.hs_s * (sx - turn), vy = 2.f * fabsf(fdy) * p.hs_s * (sy - turn);
            int fl = vy >= vx ? AF_Y : 0;
            // (the margin covers FP32 rounding of the coordinates; a range that is
            // not finite compares false)
            if (!(fmaxf(vx, vy) >= 1.01f && fminf(nT, nR) >= p.series_rmin)) fl |= AF_SLOW;
            rc[F_FLAGS] = __int_as_float(fl);
        }
        __syncwarp();
        for (int j = 0; j < cnt; ++j) {
            const float4* rc = reinterpret_cast<const float4*>(rec + j * AREC);
            const float4 r0 = rc[0], r1 = rc[1], r2 = rc[2], r3 = rc[3], r4 = rc[4], r5 = rc[5];
            const int fl = __float_as_int(r3.z);
            const bool ay = fl & AF_Y;
            const float dA = ay ? fdy : fdx, dB = ay ? fdx : fdy;
            const float rA = ay ? r0.y : r0.x, rB = ay ? r0.x : r0.y, tA = ay ? r2.y : r2.x, tB = ay ? r2.x : r2.y;
            const int nA = ay ? ny : nx, nB = ay ? nx : ny, strA = ay ? AIS : 1, strB = ay ? 1 : AIS;
            const float phk = fmaf(-r1.y, p.ph_hs, r1.z);
            if (!(fl & AF_SLOW)) {
#pragma unroll 1
                for (int l4 = 0; l4 < 4; ++l4) {
                    const int a0i = l4 & 1, b0 = (l4 >> 1) * ALINE;
                    if (a0i >= nA || b0 >= nB) continue;
                    const dfl oA = times(2 * lane + a0i - 0.5f * (AT - 1), ay ? ddy : ddx);
                    const dfl oB = times(b0 + 0.5f * (ALINE - 1) - 0.5f * (AT - 1), ay ? ddx : ddy);
                    const LineLeg T = line_leg(tA, tB, ay ? r5.y : r5.x, ay ? r5.x : r5.y, oA, oB, r2.w, r3.x, r5.z, r5.w);
                    const LineLeg R = line_leg(rA, rB, ay ? r4.y : r4.x, ay ? r4.x : r4.y, oA, oB, r0.w, r1.x, r4.z, r4.w);
                    float pl;
                    const float ph = two_sum(T.Dh, R.Dh, pl);
                    pl = pl + (T.Dl + R.Dl);
                    // half-sample coordinate v0 and carrier phase x0 at the line's centre, the phase
                    // from whole cycles removed
                    const float v0 = fmaf(ph, p.hs_s, r1.y);
                    const float cy = __fmul_rn(ph, p.k_fc_c.x);
                    const float fr = __fsub_rn(cy, __fsub_rn(__fadd_rn(cy, FLOOR_MAGIC), FLOOR_MAGIC));
                    const float x0 = fmaf(fr + fmaf(ph, p.k_fc_c.x, -cy) + fmaf(ph, p.k_fc_c.y, pl * p.k_fc_c.x),
                                          TWO_PI_F, r1.z);
                    // the series in pixels from the line's centre (exact half-integers)
                    const dfl hB = ay ? hdx : hdy;
                    const float c1s = T.c1 + R.c1, hB2 = hB.hi * dB, hB3 = hB2 * dB;
                    const float c1 = fmaf(c1s, hB.hi, c1s * hB.lo), c2 = (T.c2 + R.c2) * hB2;
                    const float c3 = (T.c3 + R.c3) * hB3, c4 = (T.c4 + R.c4) * (hB3 * dB);
                    const float2* ip = im + (2 * lane + a0i) * strA + b0 * strB;
                    const int nb = min(ALINE, nB - b0);
                    // the lane's current row and its sums: pixels along the line often share a row
                    // (the path changes slower along it), and a row is added when it is left
                    unsigned cur = 0u;
                    float2 sum[4];
                    auto put = [&](const unsigned pos, const float2 w, const float g, const bool first) {
                        float2 a[4];
                        powers(w, g, a);
                        if (first || pos != cur) {
                            if (!first) add_row(cur, sum);
                            cur = pos;
#pragma unroll
                            for (int q = 0; q < 4; ++q) sum[q] = a[q];
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q) sum[q] = fadd2(sum[q], a[q]);
                        }
                        __syncwarp();
                    };
                    float2 y = make_float2(-0.5f * (ALINE - 1), 1.f - 0.5f * (ALINE - 1));
#pragma unroll 2
                    for (int k = 0; k < nb; k += 2) {
                        // along the line from its centre: dv half samples, phase x0 + dv ph_hs
                        float2 dv = ffma2(make_float2(c4, c4), y, make_float2(c3, c3));
                        dv = ffma2(dv, y, make_float2(c2, c2));
                        dv = fmul2(ffma2(dv, y, make_float2(c1, c1)), y);
                        y = fadd2(y, make_float2(2.f, 2.f));
                        // (reduced: unreduced phases cost the SFU 1.5e-7 of their size, 1e-5 here)
                        const float2 x = reduce_phase2(ffma2(dv, make_float2(p.ph_hs, p.ph_hs), make_float2(x0, x0)));
                        const float2 v = fadd2(dv, make_float2(v0, v0));
                        const float2 t = fadd2(v, magic2), g = fsub2(v, fsub2(t, magic2));
                        const float2 I0 = ip[0], I1 = ip[strB];      // (zero past the tile's last pixel)
                        ip += 2 * strB;
                        const float2 w0 = weighted(x.x, I0), w1 = weighted(x.y, I1);
                        put(row_of(t.x), w0, g.x, k == 0);
                        put(row_of(t.y), w1, g.y, false);
                    }
                    add_row(cur, sum);
                    __syncwarp();
                }
            } else {
                for (int a = lane; a - lane < nA; a += 32) {
                    const float oA = (a - 0.5f * (AT - 1)) * dA;
                    for (int b = 0; b < nB; ++b) {
                        const float oB = (b - 0.5f * (AT - 1)) * dB, d2 = fmaf(oA, oA, oB * oB);
                        const float dR = leg_exact<false>(rB, 0.f, r0.w, r1.x, rA * oA, oB, d2);
                        const float dT = leg_exact<false>(tB, 0.f, r2.w, r3.x, tA * oA, oB, d2);
                        const float v = fmaf(dR + dT, p.hs_s, r1.y);
                        const float x = reduce_phase(fmaf(v, p.ph_hs, phk));
                        const float t = __fadd_rn(v, FLOOR_MAGIC), g = v - __fadd_rn(t, -FLOOR_MAGIC);
                        const unsigned pos = row_of(t);
                        const float2 w = weighted(x, im[a * strA + b * strB]);
                        // lanes with the same row in turn
                        const int turn = __popc(__match_any_sync(0xffffffffu, pos) & ((1u << lane) - 1u));
                        const int turns = __reduce_max_sync(0xffffffffu, turn);
                        float2 s[4];
                        powers(w, g, s);
                        for (int k = 0; k <= turns; ++k) {
                            if (turn == k) add_row(pos, s);
                            __syncwarp();
                        }
                    }
                }
            }
            // transposed FIR: out[t] = sum_m sum_h sum_p coef[h][m][p] A_p[2 (t - m) + h], three
            // consecutive samples a lane (each row is read once and used for three)
            const long long base = __float_as_int(r3.w), row = qb + AW * j;
            for (int t0 = 3 * lane; t0 < p.npos + TAPS - 1; t0 += 96) {
                float2 o[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int h = 0; h < NH; ++h) {
                    float4 e[3], f[3];   // rows of positions t0 - m + (0, 1, 2)
                    auto load = [&](int n, float4& a, float4& b) {
                        const bool in = n >= 0 && n < p.npos;
                        a = in ? rows[NH * n + h] : make_float4(0.f, 0.f, 0.f, 0.f);
                        b = in ? rows[nrow + NH * n + h] : make_float4(0.f, 0.f, 0.f, 0.f);
                    };
                    load(t0 + 1, e[1], f[1]);
                    load(t0 + 2, e[2], f[2]);
#pragma unroll
                    for (int m = 0; m < TAPS; ++m) {
                        load(t0 - m, e[0], f[0]);
                        const float4 c = coef_s[h * TAPS + m];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            o[k] = ffma2(make_float2(c.x, c.x), make_float2(e[k].x, e[k].y), o[k]);
                            o[k] = ffma2(make_float2(c.y, c.y), make_float2(e[k].z, e[k].w), o[k]);
                            o[k] = ffma2(make_float2(c.z, c.z), make_float2(f[k].x, f[k].y), o[k]);
                            o[k] = ffma2(make_float2(c.w, c.w), make_float2(f[k].z, f[k].w), o[k]);
                        }
                        e[2] = e[1]; f[2] = f[1];
                        e[1] = e[0]; f[1] = f[0];
                    }
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const long long idx = base + t0 + k;
                    if (t0 + k < p.npos + TAPS - 1 && idx >= 0 && idx < Ns && (o[k].x != 0.f || o[k].y != 0.f))
                        atomicAdd(eadj + row * Ns + idx, o[k]);
                }
            }
            __syncwarp();
            for (int i = lane; i < 2 * nrow; i += 32) rows[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncwarp();
        }
        __syncwarp();   // the records are rewritten
    }
}

}  // namespace core

// the rule for adjoint2d_kernel: straight stop-and-hop legs in 2D without a beam
// (its tiles differ from the forward pass's, so beam decisions would not agree bit
// for bit).  The accumulator rows of its eight warps take 150 KB at the
// coarsest pixel spacing prepare() takes.  Sets the launch's parameters in S.
static bool adjoint2d_plan(sas_geometry_t h, const sas_grid& g, core::Setup& S, size_t& smem) {
    using namespace core;
    KParams& p = S.prm;
    if (g.nz > 1 || p.refract || p.beam || p.vel) return false;
    const double hx = 0.5 * (AT - 1) * std::fabs(g.dx), hy = 0.5 * (AT - 1) * std::fabs(g.dy);
    const double dmax = std::sqrt(hx * hx + hy * hy);
    const int U = (int)std::ceil(2.0 * dmax * h->sig.fs / h->sig.c) + 2;
    smem = adjoint2d_smem(2 * U + 1);
    if (smem > 200 * 1024) return false;
    p.U = U;
    p.npos = 2 * U + 1;
    p.hx = (float)hx;
    p.hy = (float)hy;
    const double ymax = 0.5 * (ALINE - 1) * std::max(std::fabs(g.dx), std::fabs(g.dy));
    p.series_rmin = (float)series_range(h, dmax, ymax);
    p.tiles_x = (g.nx + AT - 1) / AT;
    p.tiles_y = (g.ny + AT - 1) / AT;
    // (loading a tile and clearing the rows costs about four pairs' time)
    const long long ntiles = (long long)p.tiles_x * p.tiles_y;
    p.pings_per_split = pick_pings_per_split(ntiles, h->P, h->C, 2LL * sm_count(), false, 4.0, 0.0, 4864);
    p.nsplit = (h->P + p.pings_per_split - 1) / p.pings_per_split;
    S.blocks = (int)(ntiles * p.nsplit);
    return true;
}

static int launch_linear_adjoint(sas_geometry_t h, const sas_grid& g, const float2* img, float2* eadj,
                                 cudaStream_t st) {
    const int dim3 = g.nz > 1;
    core::Setup S;
    int rc = core::prepare(h, g, dim3, 2LL * sm_count(), S, false);
    if (rc != SAS_OK) return rc;
    SAS_CUDA(cudaMemsetAsync(eadj, 0, sizeof(float2) * (size_t)h->P * h->C * h->Ns, st));
    size_t smem2d = 0;
    if (adjoint2d_plan(h, g, S, smem2d)) {
        SAS_CUDA(cudaFuncSetAttribute(core::adjoint2d_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2d));
        core::adjoint2d_kernel<<<S.blocks, 32 * core::AW, smem2d, st>>>(S.prm, img, eadj, h->Ns);
        SAS_CUDA(cudaGetLastError());
        return SAS_OK;
    }
    const int krec = S.prm.refract ? (int)core::NREC_REFR : (int)core::NREC;
    const size_t smem = sizeof(float2) * core::GROUP * NH * S.prm.npos * NP + sizeof(float) * krec * core::PAIRS +
                        sizeof(float) * NH * TAPS * NP + 2 * sizeof(int) * core::PAIRS;
    auto k = dim3 ? (S.prm.refract ? core::adjoint_kernel<true, true> : core::adjoint_kernel<true, false>)
                  : (S.prm.refract ? core::adjoint_kernel<false, true> : core::adjoint_kernel<false, false>);
    SAS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k<<<S.blocks, core::NTHREADS, smem, st>>>(S.prm, img, eadj, h->Ns);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

int launch_adjoint(const AdjointArgs& a) {
    if (a.grad_offsets) {
        int rc = launch_offset_grad(a.h, a.grid, a.grad_image, a.grad_offsets, a.stream);
        if (rc != SAS_OK) return rc;
    }
    if (a.echo_adj) return launch_linear_adjoint(a.h, a.grid, a.grad_image, a.echo_adj, a.stream);
    return SAS_OK;
}

}  // namespace sas

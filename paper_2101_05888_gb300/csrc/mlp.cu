// Learned fractional-delay interpolator: an MLP 1 -> 64 -> 64 -> 8 (GELU,
// FP16-stored weights, FP32 arithmetic) mapping the fractional sample
// position f to the 8 taps at offsets -3 .. 4 from floor(u), trained to
// reproduce a 32-tap Kaiser-windowed-sinc interpolation of echo windows, then
// tabulated for the backprojection kernels (which use it through the same
// interpolator slot as the Kaiser-sinc; the paper itself names no
// interpolator).
//
// Network (x = 2 f - 1):  a1 = gelu(W1 x + b1), a2 = gelu(W2 a1 + b2), t = W3 a2 + b3,
// gelu(z) = z/2 (1 + erf(z / sqrt 2)).  Loss on windows s_b (8 complex) with
// targets y_b:  L = (1/B) sum_b |sum_m t_m(f_b) s_b,m - y_b|^2.
// With a prior (the normalised 8-tap Kaiser-sinc at beta_p) the interpolator's
// taps are prior + t: the targets are the 32-tap interpolation minus the
// prior's 8-tap interpolation of the window, and the table adds the prior.
// Parameter vector (FP32 masters): W1 [64][1], b1 [64], W2 [64][64] ([out][in]),
// b2 [64], W3 [8][64], b3 [8].
#include "sas_common.cuh"

namespace sas {
namespace {

constexpr int H = 64;
constexpr int NT = 8;
constexpr int NPAR = SAS_MLP_NPARAMS;
constexpr int O_W1 = 0, O_B1 = 64, O_W2 = 128, O_B2 = 128 + 4096, O_W3 = O_B2 + 64, O_B3 = O_W3 + 512;
static_assert(O_B3 + 8 == NPAR, "parameter layout");

constexpr int SPB = 64;      // samples per block in the loss/gradient kernel
constexpr int TPB = 256;

__device__ __forceinline__ float fp16_round(float v) { return __half2float(__float2half_rn(v)); }

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

// ---------------------------------------------------------------------------
// Training windows and 32-tap Kaiser-sinc targets (FP64 weights).

__device__ double i0_series_d(double x) {
    const double q = 0.25 * x * x;
    double term = 1.0, sum = 1.0;
    for (int m = 1; m < 200; ++m) {
        term *= q / ((double)m * (double)m);
        sum += term;
        if (term < 1e-17 * sum) break;
    }
    return sum;
}

// Normalised Kaiser-windowed sinc of NTAPS taps at offsets k = 1 - NTAPS/2 .. NTAPS/2
// from floor(u), for the fraction f (FP64).
template <int NTAPS>
__device__ void kaiser_taps(double f, double beta, double* w) {
    const double h = 0.5 * NTAPS, i0b = i0_series_d(beta);
    double sum = 0.0;
    for (int m = 0; m < NTAPS; ++m) {
        const double d = f - (double)(m - NTAPS / 2 + 1);
        double v = 0.0;
        if (fabs(d) < h) {
            const double sinc = (d == 0.0) ? 1.0 : sin(M_PI * d) / (M_PI * d);
            v = sinc * i0_series_d(beta * sqrt(1.0 - (d / h) * (d / h))) / i0b;
        }
        w[m] = v;
        sum += v;
    }
    for (int m = 0; m < NTAPS; ++m) w[m] /= sum;
}

__global__ void make_windows_kernel(const float2* __restrict__ echo, int rows, int Ns, const float* __restrict__ frac,
                                    const int32_t* __restrict__ row, const int32_t* __restrict__ pos, long long n,
                                    double beta, double prior_beta, float2* __restrict__ win,
                                    float2* __restrict__ tgt) {
    const long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (b >= n) return;
    const int r = min(max(row[b], 0), rows - 1);
    const long long p0 = pos[b];
    const float2* e = echo + (size_t)r * Ns;
    for (int m = 0; m < NT; ++m) {
        const long long j = p0 + m - 3;
        win[b * NT + m] = (j >= 0 && j < Ns) ? e[j] : make_float2(0.f, 0.f);
    }
    // 32 taps k = -15 .. 16, normalised Kaiser-windowed sinc at distance f - k
    const double f = (double)frac[b];
    double w[32];
    kaiser_taps<32>(f, beta, w);
    double yr = 0.0, yi = 0.0;
    for (int m = 0; m < 32; ++m) {
        const long long j = p0 + m - 15;
        if (j < 0 || j >= Ns) continue;
        yr += w[m] * (double)e[j].x;
        yi += w[m] * (double)e[j].y;
    }
    if (prior_beta >= 0.0) {
        // residual target: less the prior's 8-tap interpolation of the window
        double wp[NT];
        kaiser_taps<NT>(f, prior_beta, wp);
        for (int m = 0; m < NT; ++m) {
            const long long j = p0 + m - 3;
            if (j < 0 || j >= Ns) continue;
            yr -= wp[m] * (double)e[j].x;
            yi -= wp[m] * (double)e[j].y;
        }
    }
    tgt[b] = make_float2((float)yr, (float)yi);
}

// ---------------------------------------------------------------------------
// Loss and gradient: each block handles SPB samples and writes its partial
// gradient; a second kernel adds the partials in block order.
//
// The three 64 x 64 x 64 products of a block (layer 2, its weight gradient, the
// gradient of layer 1's activations) run on 4 x 4 register tiles: a thread owns 4
// samples (or rows) and 4 units and reads one float4 of each operand per 16 FMAs, where
// one output a thread read two scalars per FMA and was bound by the shared-memory
// pipe (8192 samples: 36 us, now 13 us).  Every sum runs in the same order as before.
// gelu' of both layers stays in the registers of the tile's owner.

constexpr int LD = SPB + 4;      // row stride of the shared arrays: 16-byte rows, spread over the banks
static_assert(SPB == H && TPB == (SPB / 4) * (H / 4), "one 4 x 4 tile a thread");

struct MlpShared {
    float W[NPAR];               // weights rounded to FP16
    float W2T[H][LD];            // [in][out]
    float T[H][LD];              // a1 [unit][sample], then dz2 [unit][sample]
    float A1[SPB][LD];           // a1 [sample][unit]
    float A2[SPB][LD];           // a2 [sample][unit], then dz1
    float Z2[SPB][LD];           // dz2 [sample][unit]
    float DT[SPB][NT];           // dL/dt
    float X[SPB], loss[SPB], red[2];
};

// gelu(z) and gelu'(z)
__device__ __forceinline__ float gelu_both(float z, float& grad) {
    const float e = 1.0f + erff(z * 0.70710678118654752f);
    grad = 0.5f * e + z * expf(-0.5f * z * z) * 0.39894228040143268f;
    return 0.5f * z * e;
}

// acc[r][c] += sum_k a[k][r] b[k][c] over the rows k of two arrays (float4 a row of each)
__device__ __forceinline__ void tile_product(float acc[4][4], const float* a, const float* b, int ld) {
#pragma unroll 8
    for (int k = 0; k < H; ++k) {
        const float4 u = *reinterpret_cast<const float4*>(a + k * LD), v = *reinterpret_cast<const float4*>(b + k * ld);
        const float ur[4] = {u.x, u.y, u.z, u.w}, vc[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(vc[c], ur[r], acc[r][c]);
    }
}

__global__ void __launch_bounds__(TPB, 2) mlp_block_kernel(const float* __restrict__ theta, const float* __restrict__ frac,
                                                           const float2* __restrict__ win, const float2* __restrict__ tgt,
                                                           long long n, float* __restrict__ part_grad,
                                                           float* __restrict__ part_loss) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpShared& S = *reinterpret_cast<MlpShared*>(mlp_smem);
    const int tid = threadIdx.x;
    const int u0 = 4 * (tid & 15), q0 = 4 * (tid >> 4);       // the thread's units and samples
    const long long s0 = (long long)blockIdx.x * SPB;
    const int ns = (int)min((long long)SPB, n - s0);
    const float invB = 1.0f / (float)n;

    for (int k = tid; k < NPAR; k += TPB) {
        const float w = fp16_round(theta[k]);
        S.W[k] = w;
        if (k >= O_W2 && k < O_B2) S.W2T[(k - O_W2) % H][(k - O_W2) / H] = w;
    }
    if (tid < SPB) S.X[tid] = tid < ns ? 2.0f * frac[s0 + tid] - 1.0f : 0.0f;
    __syncthreads();
    // layer 1
    float g1[4][4], g2[4][4], acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float a = gelu_both(fmaf(S.W[O_W1 + u0 + c], S.X[q0 + r], S.W[O_B1 + u0 + c]), g1[r][c]);
            S.A1[q0 + r][u0 + c] = a;
            S.T[u0 + c][q0 + r] = a;
        }
    __syncthreads();
    // layer 2
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = S.W[O_B2 + u0 + c];
    tile_product(acc, &S.T[0][q0], &S.W2T[0][u0], LD);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) S.A2[q0 + r][u0 + c] = gelu_both(acc[r][c], g2[r][c]);
    __syncthreads();
    // output taps (four lanes a sample, two taps each), residual and dL/dt
    {
        const int s = tid >> 2, m0 = 2 * (tid & 3);
        float v[NT], v0 = S.W[O_B3 + m0], v1 = S.W[O_B3 + m0 + 1];
        const float *w0 = &S.W[O_W3 + m0 * H], *w1 = w0 + H;
#pragma unroll 8
        for (int i = 0; i < H; ++i) {
            const float a = S.A2[s][i];
            v0 = fmaf(w0[i], a, v0);
            v1 = fmaf(w1[i], a, v1);
        }
#pragma unroll
        for (int m = 0; m < NT; m += 2) {
            v[m] = __shfl_sync(0xffffffffu, v0, m / 2, 4);
            v[m + 1] = __shfl_sync(0xffffffffu, v1, m / 2, 4);
        }
        float rx = 0.f, ry = 0.f, d0 = 0.f, d1 = 0.f;
        if (s < ns) {
            const float2* wv = win + (s0 + s) * NT;
            rx = -tgt[s0 + s].x;
            ry = -tgt[s0 + s].y;
#pragma unroll
            for (int m = 0; m < NT; ++m) {
                const float2 w = wv[m];
                rx = fmaf(v[m], w.x, rx);
                ry = fmaf(v[m], w.y, ry);
            }
            const float2 wa = wv[m0], wb = wv[m0 + 1];
            d0 = 2.0f * invB * (rx * wa.x + ry * wa.y);   // 2/B Re(conj(r) s_m)
            d1 = 2.0f * invB * (rx * wb.x + ry * wb.y);
        }
        S.DT[s][m0] = d0;
        S.DT[s][m0 + 1] = d1;
        if (m0 == 0) S.loss[s] = rx * rx + ry * ry;
    }
    __syncthreads();
    // block loss
    if (tid < SPB) {
        float l = S.loss[tid];
        for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if ((tid & 31) == 0) S.red[tid >> 5] = l;
    }
    float* pg = part_grad + (size_t)blockIdx.x * NPAR;
    // dW3, db3
    for (int k = tid; k < NT * H + NT; k += TPB) {
        float g = 0.f;
        if (k < NT * H) {
            const int m = k / H, i = k % H;
            for (int s = 0; s < ns; ++s) g = fmaf(S.DT[s][m], S.A2[s][i], g);
            pg[O_W3 + k] = g;
        } else {
            for (int s = 0; s < ns; ++s) g += S.DT[s][k - NT * H];
            pg[O_B3 + k - NT * H] = g;
        }
    }
    // dz2 = (W3^T dt) * gelu'(z2)
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float d = 0.f;
#pragma unroll
            for (int m = 0; m < NT; ++m) d = fmaf(S.W[O_W3 + m * H + u0 + c], S.DT[q0 + r][m], d);
            d = d * g2[r][c];
            S.Z2[q0 + r][u0 + c] = d;
            S.T[u0 + c][q0 + r] = d;
        }
    __syncthreads();
    if (tid == 0) part_loss[blockIdx.x] = (S.red[0] + S.red[1]) * invB;
    // dW2 [out q0 ..][in u0 ..] over the samples (rows past ns are zero), db2
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
    tile_product(acc, &S.Z2[0][q0], &S.A1[0][u0], LD);
#pragma unroll
    for (int r = 0; r < 4; ++r)
        *reinterpret_cast<float4*>(&pg[O_W2 + (q0 + r) * H + u0]) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    if (tid < H) {
        float g = 0.f;
        for (int s = 0; s < ns; ++s) g += S.Z2[s][tid];
        pg[O_B2 + tid] = g;
    }
    // dz1 = (W2^T dz2) * gelu'(z1)
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = 0.f;
    tile_product(acc, &S.T[0][q0], &S.W[O_W2 + u0], H);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) S.A2[q0 + r][u0 + c] = acc[r][c] * g1[r][c];
    __syncthreads();
    // dW1, db1
    if (tid < 2 * H) {
        const int j = tid % H;
        float g = 0.f;
        if (tid < H)
            for (int s = 0; s < ns; ++s) g = fmaf(S.A2[s][j], S.X[s], g);
        else
            for (int s = 0; s < ns; ++s) g += S.A2[s][j];
        pg[(tid < H ? O_W1 : O_B1) + j] = g;
    }
}

// Adds the partials in FP64: 32 parameters a block, 8 threads a parameter, each over
// every eighth partial, four loads in flight (one thread a parameter over all of them
// waited on one load after the other: 32 us for 128 partials, now 5 us).
__global__ void __launch_bounds__(256) sum_partials_kernel(const float* __restrict__ part_grad,
                                                           const float* __restrict__ part_loss, int nblocks,
                                                           float* __restrict__ grad, float* __restrict__ loss) {
    __shared__ double red[8][32];
    const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;          // the last block's lane NPAR - 32 blocks: the loss
    const bool isloss = k == NPAR;
    const float* src = isloss ? part_loss : part_grad + min(k, NPAR - 1);
    const size_t step = isloss ? 1 : NPAR;
    double g = 0.0;
    int b = sl;
    for (; b + 24 < nblocks; b += 32) {
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = src[(b + 8 * u) * step];
#pragma unroll
        for (int u = 0; u < 4; ++u) g += v[u];
    }
    for (; b < nblocks; b += 8) g += src[b * step];
    red[sl][lane] = g;
    __syncthreads();
    if (sl == 0 && k <= NPAR) {
        for (int w = 1; w < 8; ++w) g += red[w][lane];
        if (isloss)
            *loss = (float)g;
        else
            grad[k] = (float)g;
    }
}

__global__ void adam_kernel(float* __restrict__ theta, const float* __restrict__ grad, float* __restrict__ m,
                            float* __restrict__ v, int step, float lr, float b1, float b2, float eps) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= NPAR) return;
    const float g = grad[k];
    const float mk = b1 * m[k] + (1.0f - b1) * g;
    const float vk = b2 * v[k] + (1.0f - b2) * g * g;
    m[k] = mk;
    v[k] = vk;
    const float mh = mk / (1.0f - powf(b1, (float)step));
    const float vh = vk / (1.0f - powf(b2, (float)step));
    theta[k] -= lr * mh / (sqrtf(vh) + eps);
}

// One thread per fraction f = j / table_n: the prior's taps (if any) plus the network's.
__global__ void tabulate_kernel(const float* __restrict__ theta, int table_n, double prior_beta,
                                float* __restrict__ out) {
    __shared__ float W[NPAR];
    for (int k = threadIdx.x; k < NPAR; k += blockDim.x) W[k] = fp16_round(theta[k]);
    __syncthreads();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > table_n) return;
    const float x = 2.0f * ((float)j / (float)table_n) - 1.0f;
    float a1[H];
    for (int q = 0; q < H; ++q) a1[q] = gelu(fmaf(W[O_W1 + q], x, W[O_B1 + q]));
    float a2[H];
    for (int i = 0; i < H; ++i) {
        float z = W[O_B2 + i];
        for (int q = 0; q < H; ++q) z = fmaf(W[O_W2 + i * H + q], a1[q], z);
        a2[i] = gelu(z);
    }
    double wp[NT];
    if (prior_beta >= 0.0) kaiser_taps<NT>((double)j / (double)table_n, prior_beta, wp);
    for (int m = 0; m < NT; ++m) {
        float v = W[O_B3 + m];
        for (int i = 0; i < H; ++i) v = fmaf(W[O_W3 + m * H + i], a2[i], v);
        out[(size_t)j * NT + m] = prior_beta >= 0.0 ? (float)(wp[m] + (double)v) : v;
    }
}

size_t block_smem() { return sizeof(MlpShared); }

}  // namespace
}  // namespace sas

using namespace sas;

extern "C" int sas_mlp_make_windows(const void* d_echo, int32_t rows, int32_t n_samples, const float* d_frac,
                                    const int32_t* d_row, const int32_t* d_pos, int64_t n, double target_beta,
                                    double prior_beta, void* d_windows, void* d_targets, void* stream) {
    if (!d_echo || rows < 1 || n_samples < 1 || n < 0 || (n > 0 && (!d_frac || !d_row || !d_pos || !d_windows ||
                                                                     !d_targets))) {
        set_error("sas_mlp_make_windows: bad argument");
        return SAS_ERR_ARG;
    }
    if (n == 0) return SAS_OK;
    make_windows_kernel<<<(unsigned)((n + 127) / 128), 128, 0, (cudaStream_t)stream>>>(
        (const float2*)d_echo, rows, n_samples, d_frac, d_row, d_pos, n, target_beta, prior_beta,
        (float2*)d_windows, (float2*)d_targets);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

extern "C" int64_t sas_mlp_workspace_bytes(int64_t n) {
    if (n < 1) return 0;
    const int64_t nb = (n + SPB - 1) / SPB;
    return nb * (int64_t)NPAR * 4 + nb * 4 + 256;
}

extern "C" int sas_mlp_loss_grad(const float* d_theta, const float* d_frac, const void* d_windows,
                                 const void* d_targets, int64_t n, float* d_loss, float* d_grad, void* d_work,
                                 void* stream) {
    if (!d_theta || !d_frac || !d_windows || !d_targets || n < 1 || !d_loss || !d_grad || !d_work) {
        set_error("sas_mlp_loss_grad: bad argument");
        return SAS_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int nb = (int)((n + SPB - 1) / SPB);
    // from the next 16-byte boundary on (the kernel stores float4; the size's spare 256
    // bytes cover the shift, so the caller's pointer may have any alignment of a float)
    float* part_grad = (float*)(((uintptr_t)d_work + 15) & ~(uintptr_t)15);
    float* part_loss = part_grad + (size_t)nb * NPAR;
    const size_t smem = block_smem();
    SAS_CUDA(cudaFuncSetAttribute(mlp_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    mlp_block_kernel<<<nb, TPB, smem, st>>>(d_theta, d_frac, (const float2*)d_windows, (const float2*)d_targets, n,
                                            part_grad, part_loss);
    SAS_CUDA(cudaGetLastError());
    sum_partials_kernel<<<(NPAR + 1 + 31) / 32, 256, 0, st>>>(part_grad, part_loss, nb, d_grad, d_loss);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

extern "C" int sas_mlp_adam(float* d_theta, const float* d_grad, float* d_m, float* d_v, int32_t step, float lr,
                            float beta1, float beta2, float eps, void* stream) {
    if (!d_theta || !d_grad || !d_m || !d_v || step < 1) {
        set_error("sas_mlp_adam: bad argument");
        return SAS_ERR_ARG;
    }
    adam_kernel<<<(NPAR + 255) / 256, 256, 0, (cudaStream_t)stream>>>(d_theta, d_grad, d_m, d_v, step, lr, beta1,
                                                                      beta2, eps);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

extern "C" int sas_interp_tabulate_mlp(const float* d_theta, int32_t table_n, double prior_beta, float* d_table_out,
                                       void* stream) {
    if (!d_theta || !d_table_out || table_n < 1 || !(prior_beta < 50.0)) {
        set_error("sas_interp_tabulate_mlp: bad argument");
        return SAS_ERR_ARG;
    }
    tabulate_kernel<<<(table_n + 1 + 127) / 128, 128, 0, (cudaStream_t)stream>>>(d_theta, table_n, prior_beta,
                                                                               d_table_out);
    SAS_CUDA(cudaGetLastError());
    return SAS_OK;
}

// Convolution-function generator on the GPU: thesis Sec. 4.2, Algorithm "convgen".
//
// Per w-plane k (w_k = w_max (k/(K-1))^2, square-root spacing, Sec. 4.2.1):
//   1. sample taper(l) taper(m) gbar_w(l, m) on an N_k x N_k image patch covering the field of
//      view l, m in [-1/(2 du), 1/(2 du)); gbar_w = 1/g_w = exp(+j 2 pi w (n - 1)) (Sec. 2.2.1);
//      the taper is psi_0(c, eta), eta = 2 du l, c = pi S0 / 2; the eta = -1 sample (no +1
//      partner) is zero; screen samples outside l^2 + m^2 < 1 are zero;
//   2. zero-pad to M = beta N_k and take a forward FFT (cuFFT Z2Z, FP64); the result samples
//      C_w at du / beta (eq. "local:o"); centring uses the (-1)^(i+j) modulation on both sides;
//   3. normalise by C_0(0,0) (Sec. 4.2.3);
//   4. support: outermost sample with |C| > threshold (Chebyshev radius R in oversampled units,
//      S = 2 ceil(R / beta) + 1), or the prescribed support ("normal" mode, Sec. 4.2.1);
//   5. trim into beta^2 sub-kernels of S x S row-major samples: sample [i][j] of sub-kernel
//      (fv, fu) is C(beta (i - h) - fv, beta (j - h) - fu), h = (S-1)/2, rows <-> v (eq.
//      "choose"), sub-kernels ordered (fv, fu), fv, fu in (-beta/2, beta/2];
//   6. zeta = sum of real parts of each sub-kernel (eq. "sum"), in FP64 before rounding to FP32.
#include <cmath>
#include <cstdio>
#include <memory>
#include <mutex>
#include <new>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "internal.cuh"

namespace wg {

__global__ void k_taper_patch(const double* coef, int ncoef, int n_k, double* t)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_k) return;
    double eta = 2.0 * (double)(i - n_k / 2) / (double)n_k;
    t[i] = (i == 0) ? 0.0 : pswf_eval_dev(coef, ncoef, eta);
}

// n - 1 = -r^2 / (1 + sqrt(1 - r^2)), zero screen outside the unit disk
__device__ __forceinline__ double2 screen(double w, double l, double m)
{
    double r2 = l * l + m * m;
    if (!(r2 < 1.0)) return make_double2(0.0, 0.0);
    double nm1 = -r2 / (1.0 + sqrt(1.0 - r2));
    double s, c;
    sincospi(2.0 * w * nm1, &s, &c);
    return make_double2(c, s);
}

// padded patch with the centring modulation (-1)^(iu + iv)
__global__ void k_fill_plane(const double* t, int n_k, int M, double du, double w, double2* out)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)M * M) return;
    int iv = (int)(idx / M), iu = (int)(idx - (int64_t)iv * M);
    int o = M / 2 - n_k / 2;
    int pv = iv - o, pu = iu - o;
    double2 v = make_double2(0.0, 0.0);
    if (pv >= 0 && pv < n_k && pu >= 0 && pu < n_k) {
        double tt = t[pv] * t[pu];
        if (tt != 0.0) {
            double l = (2.0 * (double)(pu - n_k / 2) / (double)n_k) / (2.0 * du);
            double m = (2.0 * (double)(pv - n_k / 2) / (double)n_k) / (2.0 * du);
            double2 s = screen(w, l, m);
            v = make_double2(tt * s.x, tt * s.y);
            if ((iu + iv) & 1) v = make_double2(-v.x, -v.y);
        }
    }
    out[idx] = v;
}

// C_0(0,0) of the un-normalised FFT: sum over the patch of taper x taper x screen(w = 0)
__global__ void k_dc(const double* t, int n_k, double du, double* out)
{
    __shared__ double red[256];
    double s = 0.0;
    for (int idx = threadIdx.x; idx < n_k * n_k; idx += blockDim.x) {
        int pv = idx / n_k, pu = idx - pv * n_k;
        double tt = t[pv] * t[pu];
        double l = (2.0 * (double)(pu - n_k / 2) / (double)n_k) / (2.0 * du);
        double m = (2.0 * (double)(pv - n_k / 2) / (double)n_k) / (2.0 * du);
        s += tt * screen(0.0, l, m).x;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// Chebyshev radius (oversampled units) of the outermost sample with |C| > thr * norm
__global__ void k_support_radius(const double2* C, int M, double thr2, int* radius)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int r = -1;
    if (idx < (int64_t)M * M) {
        double2 v = C[idx];
        if (v.x * v.x + v.y * v.y > thr2) {
            int iv = (int)(idx / M), iu = (int)(idx - (int64_t)iv * M);
            r = max(abs(iv - M / 2), abs(iu - M / 2));
        }
    }
    for (int o = 16; o > 0; o >>= 1) r = max(r, __shfl_xor_sync(0xffffffffu, r, o));
    if ((threadIdx.x & 31) == 0 && r >= 0) atomicMax(radius, r);
}

// one block per sub-kernel: trim, normalise, round to float, and zeta.  The samples go where the gridder and the degridder
// read them: H = (S + 1) / 2 rows of S pairs {re, re', im, im'} (pairs.cuh), the second row past the last one zero.
__global__ void k_trim(const double2* C, int M, int beta, int S, const double* normp, float4* out,
                       double* zeta)
{
    __shared__ double red[256];
    const int sub = blockIdx.x;                      // (fv - lo) * beta + (fu - lo)
    const int lo = -((beta - 1) / 2);
    const int fv = sub / beta + lo, fu = sub % beta + lo;
    const int h = (S - 1) / 2, H = (S + 1) / 2;
    const double inv = 1.0 / *normp;
    double acc = 0.0;
    float* dst = reinterpret_cast<float*>(out + (int64_t)sub * S * H);
    for (int s = threadIdx.x; s < S * S; s += blockDim.x) {
        int i = s / S, j = s - i * S;
        int ov = beta * (i - h) - fv, ou = beta * (j - h) - fu;
        int kv = ov + M / 2, ku = ou + M / 2;
        double re = 0.0, im = 0.0;
        if (kv >= 0 && kv < M && ku >= 0 && ku < M) {
            double2 v = C[(int64_t)kv * M + ku];
            double sg = ((kv + ku) & 1) ? -inv : inv;
            re = v.x * sg;
            im = v.y * sg;
        }
        const int second = i >= H ? 1 : 0;
        float* d = dst + 4 * ((i - second * H) * S + j);
        d[second] = (float)re;
        d[2 + second] = (float)im;
        if (i == H - 1) d[1] = d[3] = 0.f;               // row S
        acc += re;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) zeta[sub] = red[0];
}

static int default_nk(int s_max)
{
    int n = 64;
    while (n < 2 * s_max) n *= 2;
    return n;
}

// the pairs as bf16 or f16: the two real parts, the two imaginary parts
__global__ void k_pairs_lp(const float4* __restrict__ src, int64_t n, int store, uint2* __restrict__ dst)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 v = src[i];
    if (store == WG_BF16) {
        reinterpret_cast<__nv_bfloat162*>(dst)[2 * i] = __floats2bfloat162_rn(v.x, v.y);
        reinterpret_cast<__nv_bfloat162*>(dst)[2 * i + 1] = __floats2bfloat162_rn(v.z, v.w);
    } else {
        reinterpret_cast<__half2*>(dst)[2 * i] = __floats2half2_rn(v.x, v.y);
        reinterpret_cast<__half2*>(dst)[2 * i + 1] = __floats2half2_rn(v.z, v.w);
    }
}

// C-1 in the order of its definition from the pairs: plane k (blockIdx.y), sample i of its beta^2 S^2.  Bits are
// copied: T is a component as stored (float: 32 bits, unsigned short: bf16 or f16).
template <typename T>
__global__ void k_samples(const T* __restrict__ pairs, const int* __restrict__ supports, const int* __restrict__ offsets,
                          const unsigned* __restrict__ poffsets, int beta2, T* __restrict__ dst)
{
    const int k = blockIdx.y, S = supports[k], H = (S + 1) / 2;
    const int64_t total = (int64_t)beta2 * S * S;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t sub = i / (S * S);
        const int s = (int)(i - sub * (S * S)), second = s >= H * S ? 1 : 0;
        const T* p = pairs + 4 * ((int64_t)poffsets[k] + sub * (S * H) + s - second * H * S) + second;
        T* d = dst + 2 * ((int64_t)offsets[k] + i);
        d[0] = p[0];
        d[1] = p[2];
    }
}

static int make_samples(Table& t, cudaStream_t s)
{
    const dim3 grid(num_sms() * 8, t.K);
    const size_t n = std::max<int64_t>(t.n_samples, 1);
    float2* data = t.data;
    void* lp = t.data_lp;
    auto release = [&]() {
        if (data != t.data) cudaFree(data);
        if (lp != t.data_lp) cudaFree(lp);
    };
    if ((!data && cudaMalloc(&data, sizeof(float2) * n) != cudaSuccess) ||
        (t.store != WG_F32 && !lp && cudaMalloc(&lp, 4 * n) != cudaSuccess)) {
        cudaGetLastError();
        release();
        return fail(WG_E_OOM, "cannot allocate the table's samples in their order (%zu)", n);
    }
    if (data != t.data) {
        k_samples<<<grid, 256, 0, s>>>(reinterpret_cast<const float*>(t.pairs), t.supports_d, t.offsets_d, t.poffsets_d,
                                       t.beta * t.beta, reinterpret_cast<float*>(data));
        count_launch();
    }
    if (lp != t.data_lp) {
        k_samples<<<grid, 256, 0, s>>>(static_cast<const unsigned short*>(t.pairs_lp), t.supports_d, t.offsets_d, t.poffsets_d,
                                       t.beta * t.beta, static_cast<unsigned short*>(lp));
        count_launch();
    }
    const cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        release();
        return cuda_fail(e, "k_samples");
    }
    t.data = data;
    t.data_lp = lp;
    return WG_OK;
}

// On a stream of its own, and in the relaxed capture mode: a stream of this thread may be being captured.
int table_samples(Table& t)
{
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    if (t.data && (t.store == WG_F32 || t.data_lp)) return WG_OK;
    cudaStreamCaptureMode capture = cudaStreamCaptureModeRelaxed;
    WG_CUDA(cudaThreadExchangeStreamCaptureMode(&capture));
    cudaStream_t s = nullptr;
    int rc = WG_OK;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) rc = cuda_fail(cudaGetLastError(), "table_info");
    if (rc == WG_OK) {
        rc = make_samples(t, s);
        cudaStreamDestroy(s);
    }
    cudaThreadExchangeStreamCaptureMode(&capture);
    return rc;
}

int table_to_host(const Table& t, float* data)
{
    const int b2 = t.beta * t.beta;
    // put in order on the device and copied at once if there is room, otherwise plane by plane and put in order here
    float2* tmp = nullptr;
    if (cudaMalloc(&tmp, sizeof(float2) * (size_t)std::max<int64_t>(t.n_samples, 1)) == cudaSuccess) {
        k_samples<<<dim3(num_sms() * 8, t.K), 256>>>(reinterpret_cast<const float*>(t.pairs), t.supports_d, t.offsets_d, t.poffsets_d,
                                                     b2, reinterpret_cast<float*>(tmp));
        count_launch();
        const cudaError_t e = cudaMemcpy(data, tmp, sizeof(float2) * (size_t)t.n_samples, cudaMemcpyDeviceToHost);
        cudaFree(tmp);
        return e == cudaSuccess ? WG_OK : cuda_fail(e, "table_copy_to_host");
    }
    cudaGetLastError();
    std::vector<float4> h;
    int64_t poff = 0;
    for (int k = 0; k < t.K; ++k) {
        const int S = t.supports[k], H = (S + 1) / 2;
        const int64_t n = (int64_t)b2 * S * H;
        h.resize(n);
        WG_CUDA(cudaMemcpy(h.data(), t.pairs + poff, sizeof(float4) * n, cudaMemcpyDeviceToHost));
        float* d = data + 2 * (int64_t)t.offsets[k];
        for (int sub = 0; sub < b2; ++sub) {
            const float4* q = h.data() + (int64_t)sub * S * H;
            for (int i = 0; i < S * H; ++i, d += 2) {
                d[0] = q[i].x;
                d[1] = q[i].z;
            }
            for (int i = 0; i < S * S - S * H; ++i, d += 2) {
                d[0] = q[i].y;
                d[1] = q[i].w;
            }
        }
        poff += n;
    }
    return WG_OK;
}

int set_table_store(Table& t, int store)
{
    if (store != WG_F32 && store != WG_BF16 && store != WG_F16) return fail(WG_E_INVALID_ARG, "unknown store dtype %d", store);
    cudaFree(t.data_lp);
    cudaFree(t.pairs_lp);
    t.data_lp = nullptr;
    t.pairs_lp = nullptr;
    t.store = WG_F32;
    if (store == WG_F32) return WG_OK;
    if (cudaMalloc(&t.pairs_lp, 8 * (size_t)std::max<int64_t>(t.n_pairs, 1)) != cudaSuccess) {
        cudaGetLastError();
        return fail(WG_E_OOM, "cannot allocate the low-precision table");
    }
    if (t.n_samples > 0) {
        k_pairs_lp<<<(unsigned)((t.n_pairs + 255) / 256), 256>>>(t.pairs, t.n_pairs, store, static_cast<uint2*>(t.pairs_lp));
        WG_LAUNCHED("k_pairs_lp");
    }
    WG_CUDA(cudaDeviceSynchronize());
    t.store = store;
    return WG_OK;
}

int free_table(Table& t)
{
    cudaFree(t.data_lp);
    cudaFree(t.pairs_lp);
    cudaFree(t.pairs);
    cudaFree(t.data);
    cudaFree(t.zeta);                              // the buffer of the small arrays
    t.data_lp = t.pairs_lp = nullptr;
    t.pairs = nullptr;
    t.data = nullptr;
    t.zeta = t.wbounds_d = nullptr;
    t.wplanes_d = nullptr;
    t.supports_d = t.offsets_d = nullptr;
    t.poffsets_d = nullptr;
    t.wbounds_f = t.zeta_f = nullptr;
    return WG_OK;
}

static int finish_layout(Table& t)
{
    t.offsets.resize(t.K);
    int64_t off = 0, poff = 0;
    std::vector<unsigned> poffsets(t.K);
    t.max_support = 0;
    for (int k = 0; k < t.K; ++k) {
        t.offsets[k] = (int)off;
        poffsets[k] = (unsigned)poff;              // at most one pair a sample: below 2^31
        poff += (int64_t)t.beta * t.beta * t.supports[k] * ((t.supports[k] + 1) / 2);
        off += (int64_t)t.beta * t.beta * t.supports[k] * t.supports[k];
        t.max_support = std::max(t.max_support, t.supports[k]);
    }
    if (off >= (int64_t)1 << 31) return fail(WG_E_OOB_SUPPORT, "kernel table has %lld samples (limit 2^31)", (long long)off);
    t.n_samples = off;
    t.n_pairs = poff;
    // nearest plane in sqrt(w): plane k is chosen when b_k <= w < b_{k+1}, with
    // b_m = w_max (t t), t = (m - 1/2) / (K - 1), m = 1..K (b_K bounds the last plane)
    std::vector<double> wb(t.K, 0.0);
    if (t.K > 1)
        for (int m = 1; m <= t.K; ++m) {
            const double tm = (m - 0.5) / (double)(t.K - 1);
            wb[m - 1] = t.w_max * (tm * tm);
        }
    // the small arrays share one buffer and one copy: [zeta][wbounds][wplanes][supports][offsets][poffsets][wbounds_f][zeta_f]
    const size_t K = t.K, nz = K * t.beta * t.beta;
    const size_t bytes = sizeof(double) * (nz + 2 * K) + sizeof(int) * 4 * K + sizeof(float) * nz;
    unsigned char* d = nullptr;
    if (cudaMalloc(&t.pairs, sizeof(float4) * std::max<int64_t>(poff, 1)) != cudaSuccess ||
        cudaMalloc(&d, bytes) != cudaSuccess) {
        cudaGetLastError();
        free_table(t);
        return fail(WG_E_OOM, "cannot allocate the kernel table (%lld samples)", (long long)off);
    }
    t.zeta = reinterpret_cast<double*>(d);
    t.wbounds_d = t.zeta + nz;
    t.wplanes_d = reinterpret_cast<float2*>(t.wbounds_d + K);
    t.supports_d = reinterpret_cast<int*>(t.wplanes_d + K);
    t.offsets_d = t.supports_d + K;
    t.poffsets_d = reinterpret_cast<unsigned*>(t.offsets_d + K);
    t.wbounds_f = reinterpret_cast<float*>(t.poffsets_d + K);
    t.zeta_f = t.wbounds_f + K;
    std::vector<unsigned char> h(sizeof(double) * 2 * K + sizeof(int) * 4 * K);
    double* hw = reinterpret_cast<double*>(h.data());
    float2* hp = reinterpret_cast<float2*>(hw + K);
    int* hs = reinterpret_cast<int*>(hp + K);
    unsigned* ho = reinterpret_cast<unsigned*>(hs + 2 * K);
    float* hf = reinterpret_cast<float*>(ho + K);
    for (size_t k = 0; k < K; ++k) {
        const float hi = (float)t.w_planes[k];
        hw[k] = wb[k];
        hp[k] = make_float2(hi, (float)(t.w_planes[k] - (double)hi));
        hs[k] = t.supports[k];
        hs[K + k] = t.offsets[k];
        ho[k] = poffsets[k];
        hf[k] = (float)wb[k];                      // round to nearest
    }
    WG_CUDA(cudaMemcpy(t.wbounds_d, h.data(), h.size(), cudaMemcpyHostToDevice));
    return WG_OK;
}

__global__ void k_zeta_f32(const double* __restrict__ z, int n, float* __restrict__ zf)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) zf[i] = (float)z[i];
}

int build_table(const wg_table_desc& d, Table& t, cudaStream_t s)
{
    const int K = d.n_wplanes, beta = d.oversample;
    t.K = K;
    t.beta = beta;
    t.s0 = d.taper_support;
    t.w_max = d.w_max;
    t.du = d.du;
    t.pswf = pswf_coefficients(M_PI * d.taper_support / 2.0);
    int n_k = d.n_k;
    if (n_k == 0) {
        if ((d.support_mode & 0xFF) == WG_SUPPORT_PRESCRIBED) {
            int smax = 1;
            for (int k = 0; k < K; ++k) smax = std::max(smax, d.supports[k]);
            n_k = default_nk(smax);
        } else {
            n_k = 256;
        }
    }
    const int M = beta * n_k;
    if ((int64_t)M * M > ((int64_t)1 << 31)) return fail(WG_E_INVALID_ARG, "beta * n_k = %d too large", M);
    // device scratch
    double *coef = nullptr, *taper = nullptr, *norm = nullptr;
    double2* plane = nullptr;
    int* radius = nullptr;
    auto cleanup = [&]() {
        cudaFree(coef); cudaFree(taper); cudaFree(norm); cudaFree(plane); cudaFree(radius);
    };
    if (cudaMalloc(&coef, sizeof(double) * t.pswf.size()) != cudaSuccess ||
        cudaMalloc(&taper, sizeof(double) * n_k) != cudaSuccess ||
        cudaMalloc(&norm, sizeof(double)) != cudaSuccess ||
        cudaMalloc(&plane, sizeof(double2) * (size_t)M * M) != cudaSuccess ||
        cudaMalloc(&radius, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        cleanup();
        return fail(WG_E_OOM, "cannot allocate the %dx%d FFT plane", M, M);
    }
    cufftHandle plan;
    if (cufftPlan2d(&plan, M, M, CUFFT_Z2Z) != CUFFT_SUCCESS) {
        cleanup();
        return fail(WG_E_CUDA, "cufftPlan2d(%d) failed", M);
    }
    cufftSetStream(plan, s);
    int rc = WG_OK;
    std::vector<double> wk(K);
    for (int k = 0; k < K; ++k) wk[k] = (K == 1) ? 0.0 : d.w_max * ((double)k / (K - 1)) * ((double)k / (K - 1));
    // w-stacking: every plane holds the w = 0 kernel; the plane values w_k stay for the correction
    t.stacking = (d.support_mode & WG_TABLE_WSTACK) != 0;
    t.w_planes = wk;
    std::vector<double> wscreen(K);
    for (int k = 0; k < K; ++k) wscreen[k] = t.stacking ? 0.0 : wk[k];
    do {
        if (cudaMemcpyAsync(coef, t.pswf.data(), sizeof(double) * t.pswf.size(), cudaMemcpyHostToDevice, s) != cudaSuccess) { rc = fail(WG_E_CUDA, "copy"); break; }
        k_taper_patch<<<(n_k + 127) / 128, 128, 0, s>>>(coef, (int)t.pswf.size(), n_k, taper);
        count_launch();
        k_dc<<<1, 256, 0, s>>>(taper, n_k, d.du, norm);
        count_launch();
        const int64_t tot = (int64_t)M * M;
        const int nb = (int)((tot + 255) / 256);
        // supports
        t.supports.assign(K, 1);
        if ((d.support_mode & 0xFF) == WG_SUPPORT_PRESCRIBED) {
            for (int k = 0; k < K; ++k) t.supports[k] = d.supports[k];
        } else {
            double nrm = 0;
            if (cudaMemcpyAsync(&nrm, norm, sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess) { rc = fail(WG_E_CUDA, "norm readback"); break; }
            const double thr2 = (d.threshold * nrm) * (d.threshold * nrm);
            for (int k = 0; k < K && rc == WG_OK; ++k) {
                k_fill_plane<<<nb, 256, 0, s>>>(taper, n_k, M, d.du, wscreen[k], plane);
                count_launch();
                if (cufftExecZ2Z(plan, plane, plane, CUFFT_FORWARD) != CUFFT_SUCCESS) { rc = fail(WG_E_CUDA, "cufftExecZ2Z"); break; }
                cudaMemsetAsync(radius, 0xff, sizeof(int), s);
                k_support_radius<<<nb, 256, 0, s>>>(plane, M, thr2, radius);
                count_launch();
                int R = -1;
                if (cudaMemcpyAsync(&R, radius, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                    cudaStreamSynchronize(s) != cudaSuccess) { rc = fail(WG_E_CUDA, "support readback"); break; }
                t.supports[k] = (R < 0) ? 1 : 2 * ((R + beta - 1) / beta) + 1;
            }
            if (rc != WG_OK) break;
        }
        for (int k = 0; k < K; ++k) {
            if (t.supports[k] < 1 || t.supports[k] % 2 == 0) { rc = fail(WG_E_INVALID_ARG, "support %d of plane %d must be odd and positive", t.supports[k], k); break; }
            if (t.supports[k] > kMaxSupport) { rc = fail(WG_E_OOB_SUPPORT, "support %d of plane %d exceeds %d", t.supports[k], k, kMaxSupport); break; }
        }
        if (rc != WG_OK) break;
        rc = finish_layout(t);
        if (rc != WG_OK) break;
        int64_t poff = 0;
        for (int k = 0; k < K; ++k) {
            k_fill_plane<<<nb, 256, 0, s>>>(taper, n_k, M, d.du, wscreen[k], plane);
            count_launch();
            if (cufftExecZ2Z(plan, plane, plane, CUFFT_FORWARD) != CUFFT_SUCCESS) { rc = fail(WG_E_CUDA, "cufftExecZ2Z"); break; }
            k_trim<<<beta * beta, 256, 0, s>>>(plane, M, beta, t.supports[k], norm, t.pairs + poff,
                                                t.zeta + (int64_t)k * beta * beta);
            count_launch();
            poff += (int64_t)beta * beta * t.supports[k] * ((t.supports[k] + 1) / 2);
        }
        if (rc != WG_OK) break;
        {
            const int nz = K * beta * beta;
            k_zeta_f32<<<(nz + 255) / 256, 256, 0, s>>>(t.zeta, nz, t.zeta_f);
            count_launch();
        }
        cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_fail(e, "conv_table_build");
    } while (0);
    cufftDestroy(plan);
    cleanup();
    if (rc != WG_OK) free_table(t);
    return rc;
}

int import_table(int K, int beta, double w_max, double du, int s0, const int* supports,
                 const double* data, const double* zeta, Table& t)
{
    t.K = K;
    t.beta = beta;
    t.s0 = s0;
    t.w_max = w_max;
    t.stacking = false;
    t.w_planes.assign(K, 0.0);
    for (int k = 0; k < K && K > 1; ++k) t.w_planes[k] = w_max * ((double)k / (K - 1)) * ((double)k / (K - 1));
    t.du = du;
    t.pswf = pswf_coefficients(M_PI * s0 / 2.0);
    t.supports.assign(supports, supports + K);
    for (int k = 0; k < K; ++k)
        if (t.supports[k] < 1 || t.supports[k] % 2 == 0 || t.supports[k] > kMaxSupport)
            return fail(WG_E_INVALID_ARG, "support %d of plane %d must be odd, in [1, %d]", t.supports[k], k, kMaxSupport);
    int rc = finish_layout(t);
    if (rc != WG_OK) return rc;
    std::unique_ptr<float4[]> h(new (std::nothrow) float4[(size_t)t.n_pairs]);
    if (!h) {
        free_table(t);
        return fail(WG_E_OOM, "host allocation failed");
    }
    float4* p = h.get();
    for (int k = 0; k < K; ++k) {
        const int S = t.supports[k], n = S * ((S + 1) / 2), both = S * S - n;
        for (int sub = 0; sub < beta * beta; ++sub, p += n, data += 2 * S * S) {
            const double* q = data + 2 * n;              // the samples of the second rows
            for (int i = 0; i < both; ++i)
                p[i] = make_float4((float)data[2 * i], (float)q[2 * i], (float)data[2 * i + 1], (float)q[2 * i + 1]);
            for (int i = both; i < n; ++i) p[i] = make_float4((float)data[2 * i], 0.f, (float)data[2 * i + 1], 0.f);
        }
    }
    std::vector<float> zf((size_t)K * beta * beta);
    for (size_t i = 0; i < zf.size(); ++i) zf[i] = (float)zeta[i];
    if (cudaMemcpy(t.pairs, h.get(), sizeof(float4) * (size_t)t.n_pairs, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(t.zeta, zeta, sizeof(double) * K * beta * beta, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(t.zeta_f, zf.data(), sizeof(float) * zf.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        free_table(t);
        return fail(WG_E_CUDA, "table upload failed");
    }
    return WG_OK;
}

}  // namespace wg

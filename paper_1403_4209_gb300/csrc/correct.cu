// Image finaliser (thesis Sec. 4.7, Algorithm "finalizer") for one grid:
//   1. inverse FFT of each polarised grid, of which the images keep the real part.  The real part of the
//      inverse transform of G is the inverse transform of G's Hermitian part (G(k) + conj G(-k)) / 2, so
//      k_hermitian writes that part's half plane and cuFFT's complex-to-real transform (FP32) does half
//      the work of a complex one on half the bytes.  The Stokes images are real parts of linear
//      combinations of the polarised images, so they are combined there too, before the transform: Stokes I takes
//      one transform, not two.  Channels go in groups sized to a 1 GiB scratch.  Centring (u = 0 at
//      N/2 -> l = 0 at N/2) uses the (-1)^(x+y) modulation before and (-1)^(mx+my) after the
//      transform (N even);
//   2. division by the normaliser N_p (eq. "normalizer"); Stokes I as the mean of polarisations 0 and P-1;
//   3. divided by the taper psi_0(c, 2 du l) psi_0(c, 2 du m) (eq. "convgrid");
//   4. divided by sinc(pi l du / beta) sinc(pi m du / beta) (eq. "coversampled"),
//      with l = (k - N/2) / (N du), so 2 du l = 2 (k - N/2) / N and pi l du / beta =
//      pi (k - N/2) / (N beta).
// The divisions are multiplications by reciprocals prepared once in FP64 and applied in FP32.
// A polarisation whose normaliser is zero (no data) gives a zero image.
// WG_IMAGE_STOKES_LINEAR / _CIRCULAR combine the polarisations, each divided by its own N_p, into I, Q, U, V
// (step 2 "convert to multiple-Stokes image and normalise").
// WG_IMAGE_WSTACK sums the planes of each channel after their (complex) inverse FFTs, each multiplied by its
// exp(+j2pi w_k (n-1)) (eq. "stacking"), then takes steps 2-4 with the channel's N_p.
// What bounds it: HBM, and the transforms' own passes.  Measured (grid_correct): Stokes I of 16 channels of 2048^2 x 4
// 1.93 -> 0.78 ms; of 4 channels of 8192^2 x 1 5.24 -> 2.29 ms; I, Q, U, V of 3 channels of 1500^2 569 -> 428 us; w-stacking of
// 32 planes of 2048^2 x 1 3.72 -> 1.36 ms (32 launches that each read and wrote the sums, and FP64 phases, before).
// WG_IMAGE_PER_POL_RAW skips the division by N_p.  It images the residuals of a fit to visibilities, and at sides that are
// powers of two it keeps complex transforms: of these smooth, peaked grids cuFFT's complex-to-real ones came out less
// accurate there (rel-L2 against 64 bits 3.1e-7 against 2.5e-7 at 1024^2, and 3.2e-7 against 2.5e-7 at 2048^2; the gradient of a
// fit at 1024^2 4.4e-7 against 3.4e-7), at other sides as accurate or more so (gradients 3.4e-7 against 4.1e-7 at 896^2, 3.6
// against 3.8 at 1152^2, 2.6 against 2.8 at 1500^2).  Of gridded observations they are as accurate (1024^2: 3.2e-7 against
// 3.1e-7) or more so (512^2 2.2 against 2.6, 1500^2 2.5 against 2.9, 2048^2 2.7 against 3.1, 8192^2 3.3 against 3.6).
// WG_IMAGE_TRANSPOSE applies the exact transpose
// of that map (the adjoint of Re(inverse FFT) under the real inner product is the forward FFT of
// the real image): grid = (-1)^(x+y) FFT_forward((-1)^(mx+my) img / (taper sinc)), a real-to-complex
// transform whose other half plane k_expand mirrors into the grid.
#include "internal.cuh"

namespace wg {

__global__ void k_corr_vec(const double* __restrict__ coef, int ncoef, int N, int beta, double* __restrict__ corr,
                           float* __restrict__ icorr)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    const double eta = 2.0 * (double)(k - N / 2) / (double)N;
    const double t = pswf_eval_dev(coef, ncoef, eta);
    const double x = M_PI * (double)(k - N / 2) / ((double)N * beta);
    const double sn = (x == 0.0) ? 1.0 : sin(x) / x;
    corr[k] = t * sn;
    icorr[k] = (float)(1.0 / (t * sn));
}

// 1 / N_p, or 0 where a polarisation has no data
__device__ __forceinline__ float inv_norm(double n) { return n != 0.0 ? (float)(1.0 / n) : 0.f; }

// The polarisations of one pixel as the mode's images take them (linear combinations; step 2 for Stokes).
// NO images: the P polarisations, or Stokes I alone.  in: the reciprocals of N_p.
template <int P, int NO>
__device__ __forceinline__ void combine(const float2 (&g)[P], const float (&in)[P], int mode, float2 (&o)[NO])
{
    if constexpr (NO == 1 && P > 1) {          // Stokes I
        o[0] = make_float2(0.5f * (g[0].x * in[0] + g[P - 1].x * in[P - 1]), 0.5f * (g[0].y * in[0] + g[P - 1].y * in[P - 1]));
    } else if (P == 1 || (mode != WG_IMAGE_STOKES_LINEAR && mode != WG_IMAGE_STOKES_CIRCULAR)) {
#pragma unroll
        for (int p = 0; p < NO; ++p) o[p] = g[p];     // scaled after the transform
    } else {
        float2 z[P];
#pragma unroll
        for (int p = 0; p < P; ++p) z[p] = make_float2(g[p].x * in[p], g[p].y * in[p]);
        auto half_sum = [](float2 a, float2 b) { return make_float2(0.5f * (a.x + b.x), 0.5f * (a.y + b.y)); };
        auto half_dif = [](float2 a, float2 b) { return make_float2(0.5f * (a.x - b.x), 0.5f * (a.y - b.y)); };
        if constexpr (P == 2) {
            o[0] = half_sum(z[0], z[1]);       // I
            o[1] = half_dif(z[0], z[1]);       // Q = (XX - YY)/2, or V = (RR - LL)/2
        } else if constexpr (P == 4) {
            const float2 crs = half_dif(z[1], z[2]);
            o[0] = half_sum(z[0], z[3]);       // I
            const float2 par_d = half_dif(z[0], z[3]), crs_s = half_sum(z[1], z[2]), crs_d = make_float2(crs.y, -crs.x);
            if (mode == WG_IMAGE_STOKES_LINEAR) {
                o[1] = par_d;                  // Q = (XX - YY)/2
                o[2] = crs_s;                  // U = (XY + YX)/2
                o[3] = crs_d;                  // V = -j (XY - YX)/2
            } else {
                o[1] = crs_s;                  // Q = (RL + LR)/2
                o[2] = crs_d;                  // U = -j (RL - LR)/2
                o[3] = par_d;                  // V = (RR - LL)/2
            }
        }
    }
}

template <int P>
__device__ __forceinline__ void load_pix(const float2* __restrict__ g, float2 (&v)[P])
{
    if constexpr (P == 1) {
        v[0] = g[0];
    } else {
#pragma unroll
        for (int h = 0; h < P; h += 2) {
            const float4 a = *reinterpret_cast<const float4*>(g + h);
            v[h] = make_float2(a.x, a.y);
            v[h + 1] = make_float2(a.z, a.w);
        }
    }
}

// step 1 input for a group of channels: of each image's combination, times (-1)^(x+y), the Hermitian part's half
// plane f[o][gch][N][N/2 + 1].  Thread: (x, y = blockIdx.y, channel = blockIdx.z).  HBM-bound: every pixel is read once.
template <int P, int NO>
__global__ void __launch_bounds__(256) k_hermitian(const float2* __restrict__ grid, const double* __restrict__ norm,
                                                   float2* __restrict__ f, int N, int mode)
{
    __shared__ float s_in[P];
    const int y = blockIdx.y, gch = blockIdx.z, G = gridDim.z, M = N / 2 + 1;
    if (threadIdx.x < P) s_in[threadIdx.x] = mode == WG_IMAGE_PER_POL_RAW ? 1.f : inv_norm(norm[gch * P + threadIdx.x]);
    __syncthreads();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= M) return;
    float in[P];
#pragma unroll
    for (int p = 0; p < P; ++p) in[p] = s_in[p];
    const float2* gc = grid + (size_t)gch * N * N * P;
    const int ym = y ? N - y : 0, xm = x ? N - x : 0;
    float2 a[P], b[P], oa[NO], ob[NO];
    load_pix<P>(gc + ((size_t)y * N + x) * P, a);
    load_pix<P>(gc + ((size_t)ym * N + xm) * P, b);
    combine<P, NO>(a, in, mode, oa);
    combine<P, NO>(b, in, mode, ob);
    const float sg = ((x + y) & 1) ? -0.5f : 0.5f;
#pragma unroll
    for (int o = 0; o < NO; ++o)
        f[(((size_t)o * G + gch) * N + y) * M + x] = make_float2(sg * (oa[o].x + ob[o].x), sg * (oa[o].y - ob[o].y));
}

// steps 2-4 from the real planes r[o][gch][N][N] to the images [gch][o][N][N], two pixels a thread
// (blockIdx.y = row, blockIdx.z = gch * NO + o); scaled: the mode's images are still to be divided by N_p
__global__ void __launch_bounds__(256) k_finish_planes(const float* __restrict__ r, int N, int P, int NO, int G,
                                                       const float* __restrict__ icorr, const double* __restrict__ norm,
                                                       int scaled, float* __restrict__ img)
{
    __shared__ float s_row;
    const int my = blockIdx.y, gch = blockIdx.z / NO, o = blockIdx.z - gch * NO;
    if (threadIdx.x == 0) s_row = icorr[my] * (scaled ? inv_norm(norm[gch * P + o]) : 1.f) * ((my & 1) ? -1.f : 1.f);
    __syncthreads();
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x >= N) return;
    const float2 v = *reinterpret_cast<const float2*>(r + (((size_t)o * G + gch) * N + my) * N + x);
    const float2 c = *reinterpret_cast<const float2*>(icorr + x);
    float* d = img + ((size_t)blockIdx.z * N + my) * N + x;
    const float a = v.x * (c.x * s_row), b = -v.y * (c.y * s_row);
    if ((reinterpret_cast<uintptr_t>(img) & 7) == 0) {
        *reinterpret_cast<float2*>(d) = make_float2(a, b);
    } else {                                   // an image buffer that is only float-aligned
        d[0] = a;
        d[1] = b;
    }
}

// transpose, step 1: real planes (-1)^(mx+my) img / (taper sinc), [gch][p][N][N] (blockIdx.z)
__global__ void __launch_bounds__(256) k_image_in(const float* __restrict__ img, int N, const float* __restrict__ icorr,
                                                  float* __restrict__ r)
{
    const int my = blockIdx.y, x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x >= N) return;
    const size_t at = ((size_t)blockIdx.z * N + my) * N + x;
    const float row = icorr[my] * ((my & 1) ? -1.f : 1.f);
    const float2 c = *reinterpret_cast<const float2*>(icorr + x);
    *reinterpret_cast<float2*>(r + at) = make_float2(img[at] * (c.x * row), img[at + 1] * (-c.y * row));
}

// transpose, step 3: the grid from the half planes f[gch][p][N][N/2 + 1] of the real images' transforms, times (-1)^(x+y)
template <int P>
__global__ void __launch_bounds__(256) k_expand(const float2* __restrict__ f, float2* __restrict__ grid, int N)
{
    const int y = blockIdx.y, x = blockIdx.x * blockDim.x + threadIdx.x, M = N / 2 + 1;
    if (x >= N) return;
    const bool mirror = x >= M;
    const int ys = mirror ? (y ? N - y : 0) : y, xs = mirror ? N - x : x;
    const float sx = ((x + y) & 1) ? -1.f : 1.f, sy = mirror ? -sx : sx;
    float2 v[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float2 a = f[(((size_t)blockIdx.z * P + p) * N + ys) * M + xs];
        v[p] = make_float2(sx * a.x, sy * a.y);
    }
    float2* d = grid + (((size_t)blockIdx.z * N + y) * N + x) * P;
    if constexpr (P == 1) {
        d[0] = v[0];
    } else {
#pragma unroll
        for (int h = 0; h < P; h += 2) *reinterpret_cast<float4*>(d + h) = make_float4(v[h].x, v[h].y, v[h + 1].x, v[h + 1].y);
    }
}

// the P polarisations of a group's pixels into contiguous planes f[gch][p][N][N] (P > 1)
template <int P>
__global__ void __launch_bounds__(256) k_planes(const float2* __restrict__ grid, float2* __restrict__ f, int64_t nn)
{
    const int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pix >= nn) return;
    float2 v[P];
    load_pix<P>(grid + (blockIdx.y * nn + pix) * P, v);
#pragma unroll
    for (int p = 0; p < P; ++p) f[(blockIdx.y * (int64_t)P + p) * nn + pix] = v[p];
}

// WG_IMAGE_PER_POL_RAW, N a power of two: the real parts of the planes f[gch][p][N][N] (blockIdx.z) of the inverse transforms (not
// demodulated, so that pixel m is at (m + N/2) mod N) times (-1)^(mx+my) / (taper sinc)
__global__ void __launch_bounds__(256) k_image_out(const float2* __restrict__ f, int N, const float* __restrict__ icorr,
                                                   float* __restrict__ img)
{
    const int my = blockIdx.y, x = blockIdx.x * blockDim.x + threadIdx.x, h = N / 2;
    if (x >= N) return;
    const size_t plane = (size_t)blockIdx.z * N * N;
    const float c = icorr[my] * icorr[x] * (((x + my) & 1) ? -1.f : 1.f);
    img[plane + (size_t)my * N + x] = f[plane + (size_t)(my >= h ? my - h : my + h) * N + (x >= h ? x - h : x + h)].x * c;
}

// w-stacking (eq. "stacking"): n - 1 over one quadrant of the image (it depends on |l| and |m|), as the sum of two
// floats; NaN outside the unit disk (l^2 + m^2 >= 1)
__global__ void k_nm1(int M, int N, double du, float2* __restrict__ nm1)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= M) return;
    const double l = (double)i / ((double)N * du), m = (double)j / ((double)N * du);
    const double r2 = l * l + m * m;
    const double v = (r2 < 1.0) ? -r2 / (1.0 + sqrt(1.0 - r2)) : __longlong_as_double(0x7FF8000000000000ll);
    const float hi = (float)v;
    nm1[(size_t)j * M + i] = make_float2(hi, (float)(v - (double)hi));
}

// Adds the planes [g0, g1) of input channel c (grid channels c K + k; f holds the inverse FFTs of grid channels from c0 on,
// not demodulated, so that pixel m is at (m + N/2) mod N) to its images: sum of Re(f exp(+j 2 pi w_k (n - 1))), the
// only part the images keep.  The phase is reduced exactly: w_k (n - 1) in two floats (FMA), its integer part
// off the high one.  One pass over all planes of a group with the sums in registers; the last
// group's sums are finished (steps 2-4).  blockIdx.y = row, blockIdx.z = input channel - cin0.
template <int P>
__global__ void __launch_bounds__(256) k_stack(const float2* __restrict__ f, int N, int K, int c0, int c1, int cin0,
                                               const float2* __restrict__ nm1, const float2* __restrict__ wpl,
                                               const float* __restrict__ icorr, const double* __restrict__ norm,
                                               float* __restrict__ img)
{
    const int mx = blockIdx.x * blockDim.x + threadIdx.x, my = blockIdx.y, c = cin0 + blockIdx.z, h = N / 2;
    if (mx >= N) return;
    const int g0 = max(c0, c * K), g1 = min(c1, (c + 1) * K);
    const size_t nn = (size_t)N * N;
    float* out = img + (size_t)c * P * nn + (size_t)my * N + mx;
    float acc[P];
#pragma unroll
    for (int p = 0; p < P; ++p) acc[p] = g0 == c * K ? 0.f : out[p * nn];
    const float2 v = nm1[(size_t)abs(my - h) * (h + 1) + abs(mx - h)];
    if (v.x == v.x) {                                   // inside the unit disk (the screen is 0 outside)
        const float2* src = f + (size_t)(g0 - c0) * P * nn + (size_t)(my >= h ? my - h : my + h) * N + (mx >= h ? mx - h : mx + h);
        for (int g = g0; g < g1; ++g, src += P * nn) {
            const float2 w = wpl[g - c * K];
            const float p0 = __fmul_rn(w.x, v.x);
            const float e = fmaf(w.x, v.x, -p0) + fmaf(w.x, v.y, w.y * v.x);
            float sn, cs;
            sincospif(2.0f * ((p0 - rintf(p0)) + e), &sn, &cs);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const float2 a = src[p * nn];
                acc[p] += a.x * cs - a.y * sn;
            }
        }
    }
    const float cc = ((mx + my) & 1 ? -1.f : 1.f) * icorr[mx] * icorr[my];
#pragma unroll
    for (int p = 0; p < P; ++p)
        out[p * nn] = g1 == (c + 1) * K ? acc[p] * cc * inv_norm(norm[(size_t)c * K * P + p]) : acc[p];
}

static int make_plan(cufftHandle& plan, int N, cufftType type, int batch)
{
    if (plan >= 0) return WG_OK;
    int n[2] = {N, N}, half[2] = {N, N / 2 + 1};
    const int full = N * N, hp = N * (N / 2 + 1);
    // a plan takes 0.3 to 0.9 ms, so each is made by the first call that needs it, also while a stream of
    // this thread is being captured: making a plan allocates, which a relaxed capture mode allows
    cudaStreamCaptureMode capture = cudaStreamCaptureModeRelaxed;
    WG_CUDA(cudaThreadExchangeStreamCaptureMode(&capture));
    cufftResult rc;
    if (type == CUFFT_C2R) rc = cufftPlanMany(&plan, 2, n, half, 1, hp, n, 1, full, type, batch);
    else if (type == CUFFT_R2C) rc = cufftPlanMany(&plan, 2, n, n, 1, full, half, 1, hp, type, batch);
    else rc = cufftPlanMany(&plan, 2, n, n, 1, full, n, 1, full, type, batch);
    cudaThreadExchangeStreamCaptureMode(&capture);
    if (rc != CUFFT_SUCCESS) {
        plan = -1;
        return fail(WG_E_CUDA, "cufftPlanMany(%d x %d, batch %d) failed", N, N, batch);
    }
    return WG_OK;
}

template <int P>
static int correct_impl(Grid& g, const Table& t, int mode, float* image, cudaStream_t s)
{
    const int N = g.n, C = g.n_chan, M = N / 2 + 1;
    const int64_t per_chan = (int64_t)N * N * P;
    if (!g.scratch) {
        // channels per group: the largest divisor of C whose grids fit in 1 GiB; the scratch holds them as complex
        // planes, or as half planes and real planes
        int G = 1;
        for (int d = 1; d <= C; ++d)
            if (C % d == 0 && (int64_t)d * per_chan * (int64_t)sizeof(float2) <= ((int64_t)1 << 30)) G = d;
        if (cudaMalloc(&g.scratch, sizeof(float2) * (size_t)G * P * N * (N + 1) + 256) != cudaSuccess ||
            cudaMalloc(&g.corr, sizeof(double) * N) != cudaSuccess ||
            cudaMalloc(&g.icorr, sizeof(float) * N) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(g.scratch);
            cudaFree(g.corr);
            g.scratch = nullptr;
            g.corr = nullptr;
            return fail(WG_E_OOM, "cannot allocate the FFT scratch grid");
        }
        g.scratch_chans = G;
    }
    const int G = g.scratch_chans;
    const bool raw_c2c = mode == WG_IMAGE_PER_POL_RAW && (N & (N - 1)) == 0;
    {
        int rc;
        if (mode == WG_IMAGE_TRANSPOSE) rc = make_plan(g.plan_r2c, N, CUFFT_R2C, G * P);
        else if (mode == WG_IMAGE_WSTACK || raw_c2c) rc = make_plan(g.plan_c2c, N, CUFFT_C2C, G * P);
        else rc = make_plan(g.plan_c2r, N, CUFFT_C2R, G);
        if (rc != WG_OK) return rc;
    }
    if (g.corr_s0 != t.s0 || g.corr_beta != t.beta) {
        double* coef = nullptr;
        WG_CUDA(cudaMalloc(&coef, sizeof(double) * t.pswf.size()));
        WG_CUDA(cudaMemcpy(coef, t.pswf.data(), sizeof(double) * t.pswf.size(), cudaMemcpyHostToDevice));
        k_corr_vec<<<(N + 127) / 128, 128, 0, s>>>(coef, (int)t.pswf.size(), N, t.beta, g.corr, g.icorr);
        WG_LAUNCHED("k_corr_vec");
        WG_CUDA(cudaStreamSynchronize(s));
        cudaFree(coef);
        g.corr_s0 = t.s0;
        g.corr_beta = t.beta;
    }
    const dim3 full((N + 255) / 256, N), half((M + 255) / 256, N), pair((N / 2 + 255) / 256, N);
    auto with_z = [](dim3 d, int z) { return dim3(d.x, d.y, (unsigned)z); };
    if (mode == WG_IMAGE_TRANSPOSE) {
        float* real = reinterpret_cast<float*>(g.scratch);
        // real planes first, the half planes behind them (256-byte aligned)
        float2* hp = g.scratch + ((size_t)G * per_chan / 2 + 31) / 32 * 32;
        if (cufftSetStream(g.plan_r2c, s) != CUFFT_SUCCESS) return fail(WG_E_CUDA, "cufftSetStream failed");
        for (int c0 = 0; c0 < C; c0 += G) {
            k_image_in<<<with_z(pair, G * P), 256, 0, s>>>(image + (size_t)c0 * per_chan, N, g.icorr, real);
            WG_LAUNCHED("k_image_in");
            if (cufftExecR2C(g.plan_r2c, real, reinterpret_cast<cufftComplex*>(hp)) != CUFFT_SUCCESS)
                return fail(WG_E_CUDA, "cufftExecR2C failed");
            k_expand<P><<<with_z(full, G), 256, 0, s>>>(hp, g.data + (size_t)c0 * per_chan, N);
            WG_LAUNCHED("k_expand");
        }
        return WG_OK;
    }
    const int64_t nn = (int64_t)N * N;
    // the inverse transforms of channels c0 .. c0 + G - 1 into the scratch, as planes, not demodulated
    auto transform = [&](int c0) -> int {
        float2* src = g.data + (size_t)c0 * per_chan;
        if constexpr (P > 1) {
            k_planes<P><<<dim3((unsigned)((nn + 255) / 256), (unsigned)G), 256, 0, s>>>(src, g.scratch, nn);
            WG_LAUNCHED("k_planes");
            src = g.scratch;
        }
        if (cufftExecC2C(g.plan_c2c, reinterpret_cast<cufftComplex*>(src), reinterpret_cast<cufftComplex*>(g.scratch),
                         CUFFT_INVERSE) != CUFFT_SUCCESS)
            return fail(WG_E_CUDA, "cufftExecC2C failed");
        return WG_OK;
    };
    if (raw_c2c) {
        if (cufftSetStream(g.plan_c2c, s) != CUFFT_SUCCESS) return fail(WG_E_CUDA, "cufftSetStream failed");
        for (int c0 = 0; c0 < C; c0 += G) {
            if (int rc = transform(c0)) return rc;
            k_image_out<<<with_z(full, G * P), 256, 0, s>>>(g.scratch, N, g.icorr, image + (size_t)c0 * per_chan);
            WG_LAUNCHED("k_image_out");
        }
        return WG_OK;
    }
    if (mode == WG_IMAGE_WSTACK) {
        const int K = t.K;
        const size_t bytes = sizeof(float2) * (size_t)M * M;
        float2* nm1 = nullptr;
        if (cudaMallocAsync((void**)&nm1, bytes, s) != cudaSuccess) {
            cudaGetLastError();
            return fail(WG_E_OOM, "cannot allocate the w-stacking screen (%zu bytes)", bytes);
        }
        int rc = WG_OK;
        k_nm1<<<dim3((M + 255) / 256, M), 256, 0, s>>>(M, N, g.du, nm1);
        count_launch();
        if (cufftSetStream(g.plan_c2c, s) != CUFFT_SUCCESS) rc = fail(WG_E_CUDA, "cufftSetStream failed");
        for (int c0 = 0; c0 < C && rc == WG_OK; c0 += G) {
            rc = transform(c0);
            const int cin0 = c0 / K, cin1 = (c0 + G - 1) / K;
            if (rc == WG_OK) {
                k_stack<P><<<with_z(full, cin1 - cin0 + 1), 256, 0, s>>>(g.scratch, N, K, c0, c0 + G, cin0, nm1, t.wplanes_d,
                                                                       g.icorr, g.norm, image);
                count_launch();
            }
        }
        if (rc == WG_OK && cudaGetLastError() != cudaSuccess) rc = fail(WG_E_CUDA, "w-stacking kernels failed to launch");
        cudaFreeAsync(nm1, s);
        return rc;
    }
    const int no = mode == WG_IMAGE_STOKES_I ? 1 : P;
    const bool scaled = mode == WG_IMAGE_PER_POL || (P == 1 && mode != WG_IMAGE_PER_POL_RAW);
    if (cufftSetStream(g.plan_c2r, s) != CUFFT_SUCCESS) return fail(WG_E_CUDA, "cufftSetStream failed");
    float2* hp = g.scratch;                    // half planes [no][G], then the real planes behind them
    float* real = reinterpret_cast<float*>(g.scratch + ((size_t)no * G * N * M + 31) / 32 * 32);
    for (int c0 = 0; c0 < C; c0 += G) {
        const float2* src = g.data + (size_t)c0 * per_chan;
        const double* norm = g.norm + (size_t)c0 * P;
        if (no == P) k_hermitian<P, P><<<with_z(half, G), 256, 0, s>>>(src, norm, hp, N, mode);
        else k_hermitian<P, 1><<<with_z(half, G), 256, 0, s>>>(src, norm, hp, N, mode);
        WG_LAUNCHED("k_hermitian");
        for (int o = 0; o < no; ++o)
            if (cufftExecC2R(g.plan_c2r, reinterpret_cast<cufftComplex*>(hp + (size_t)o * G * N * M),
                             real + (size_t)o * G * N * N) != CUFFT_SUCCESS)
                return fail(WG_E_CUDA, "cufftExecC2R failed");
        k_finish_planes<<<with_z(pair, G * no), 256, 0, s>>>(real, N, P, no, G, g.icorr, norm, scaled ? 1 : 0,
                                                            image + (size_t)c0 * no * N * N);
        WG_LAUNCHED("k_finish_planes");
    }
    return WG_OK;
}

int launch_correct(Grid& g, const Table& t, int mode, float* image, cudaStream_t s)
{
    switch (g.n_pol) {
        case 1: return correct_impl<1>(g, t, mode, image, s);
        case 2: return correct_impl<2>(g, t, mode, image, s);
        case 4: return correct_impl<4>(g, t, mode, image, s);
        default: return fail(WG_E_INVALID_ARG, "n_pol must be 1, 2 or 4");
    }
}

}  // namespace wg

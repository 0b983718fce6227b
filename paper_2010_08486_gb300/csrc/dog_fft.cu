// FFT-convolution backend of the scale space (Sec. 4.1 names FFT convolution
// as the alternative to direct convolution; Sec. 5 compares the two).
//
// Per frame: the frame is reflect-padded by R (the largest radius, with the
// same half-sample fold as the direct path) into a grid of Hp x Wp cells
// (2-3-5-7-smooth sizes, Hp >= max_h + 2R, Wp >= max_w + 2R, zeros beyond);
// one real-to-complex FFT; for every level the spectrum is multiplied by the
// level's kernel spectrum, which is real and separable (the sampled Gaussian
// is even): G_i(ky, kx) = g_i(ky) g_i(kx), g(k) = w_0 + 2 sum_t w_t cos(2 pi k
// t / N), computed in double on the host; one batched complex-to-real inverse
// FFT gives every L_i on the grid, where the frame's pixel (y, x) sits at
// (y + R, x + R) and no circular wrap reaches it (the kernels span at most R).
// A stencil kernel then forms D_l = c_l (L_l - L_{l+1}) and applies the same
// 3x3x3 test and strict threshold as the direct path, compacting candidates
// with one atomic each.  The FFTs run in single precision (cuFFT); the values
// differ from the direct sums by the transforms' rounding.
#include <cuda_runtime.h>
#include <cufft.h>

#include <cmath>
#include <vector>

#include "dog_internal.cuh"
#include "dog_device.cuh"

namespace dogk {

struct FftWS {
    int Hp = 0, Wp = 0, K = 0, R = 0;
    int last_h = 0, last_w = 0;   // frame size of the last padding (grid cells past it are zero)
    cufftHandle fwd = 0, inv = 0;
    bool have_fwd = false, have_inv = false;
    float* pad = nullptr;         // Hp x Wp
    cufftComplex* spec = nullptr; // Hp x (Wp/2+1)
    cufftComplex* specs = nullptr;  // K x Hp x (Wp/2+1)
    float* planes = nullptr;      // K x Hp x Wp
    float* gx = nullptr;          // K x (Wp/2+1) kernel spectra along x (divided by Hp Wp)
    float* gy = nullptr;          // K x Hp kernel spectra along y
};

// smallest n >= m whose prime factors are 2, 3, 5 and 7
int fft_size(int m) {
    for (int n = m > 1 ? m : 1;; ++n) {
        int v = n;
        for (int p : {2, 3, 5, 7})
            while (v % p == 0) v /= p;
        if (v == 1) return n;
    }
}

void fft_free(FftWS* f) {
    if (!f) return;
    if (f->have_fwd) cufftDestroy(f->fwd);
    if (f->have_inv) cufftDestroy(f->inv);
    void* ptrs[] = {f->pad, f->spec, f->specs, f->planes, f->gx, f->gy};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete f;
}

// Workspace and plans for frames up to max_h x max_w; kernel spectra of the
// handle's ladder (w: K kernels of 2 r_i + 1 taps, tap t weighing offset t - r).
int fft_create(FftWS** out, int max_h, int max_w, int K, int R, const std::vector<std::vector<double>>& w) {
    FftWS* f = new (std::nothrow) FftWS();
    if (!f) return DOG_ERR_NOMEM;
    f->Hp = fft_size(max_h + 2 * R);
    f->Wp = fft_size(max_w + 2 * R);
    f->K = K;
    f->R = R;
    const int Wc = f->Wp / 2 + 1;
    const size_t n_pad = (size_t)f->Hp * f->Wp, n_spec = (size_t)f->Hp * Wc;
    cudaError_t e = cudaSuccess;
    auto ok = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    ok(cudaMalloc(&f->pad, sizeof(float) * n_pad));
    ok(cudaMalloc(&f->spec, sizeof(cufftComplex) * n_spec));
    ok(cudaMalloc(&f->specs, sizeof(cufftComplex) * n_spec * K));
    ok(cudaMalloc(&f->planes, sizeof(float) * n_pad * K));
    ok(cudaMalloc(&f->gx, sizeof(float) * (size_t)K * Wc));
    ok(cudaMalloc(&f->gy, sizeof(float) * (size_t)K * f->Hp));
    if (e == cudaSuccess) ok(cudaMemset(f->pad, 0, sizeof(float) * n_pad));
    if (e != cudaSuccess) {
        fft_free(f);
        return e == cudaErrorMemoryAllocation ? DOG_ERR_NOMEM : DOG_ERR_CUDA;
    }
    // kernel spectra, double on the host, rounded to float; 1 / (Hp Wp) (the
    // inverse transform's scale) folded into gx
    std::vector<float> hx((size_t)K * Wc), hy((size_t)K * f->Hp);
    const double two_pi = 2.0 * M_PI, scale = 1.0 / ((double)f->Hp * (double)f->Wp);
    for (int i = 0; i < K; ++i) {
        const int r = ((int)w[i].size() - 1) / 2;
        for (int k = 0; k < Wc; ++k) {
            double g = w[i][r];
            for (int t = 1; t <= r; ++t) g += 2.0 * w[i][r + t] * std::cos(two_pi * (double)k * t / f->Wp);
            hx[(size_t)i * Wc + k] = (float)(g * scale);
        }
        for (int k = 0; k < f->Hp; ++k) {
            double g = w[i][r];
            for (int t = 1; t <= r; ++t) g += 2.0 * w[i][r + t] * std::cos(two_pi * (double)k * t / f->Hp);
            hy[(size_t)i * f->Hp + k] = (float)g;
        }
    }
    ok(cudaMemcpy(f->gx, hx.data(), sizeof(float) * hx.size(), cudaMemcpyHostToDevice));
    ok(cudaMemcpy(f->gy, hy.data(), sizeof(float) * hy.size(), cudaMemcpyHostToDevice));
    if (e == cudaSuccess) {
        if (cufftPlan2d(&f->fwd, f->Hp, f->Wp, CUFFT_R2C) != CUFFT_SUCCESS) e = cudaErrorUnknown;
        else f->have_fwd = true;
    }
    if (e == cudaSuccess) {
        int n[2] = {f->Hp, f->Wp};
        if (cufftPlanMany(&f->inv, 2, n, nullptr, 1, (int)n_spec, nullptr, 1, (int)n_pad, CUFFT_C2R, K) !=
            CUFFT_SUCCESS)
            e = cudaErrorUnknown;
        else
            f->have_inv = true;
    }
    if (e != cudaSuccess) {
        fft_free(f);
        return e == cudaErrorMemoryAllocation ? DOG_ERR_NOMEM : DOG_ERR_CUDA;
    }
    *out = f;
    return DOG_OK;
}

// Reflect-padded frame on the grid: cell (Y, X) for Y < H + 2R, X < W + 2R
// holds pixel (refl(Y - R), refl(X - R)); the rest of the grid stays zero.  Four
// rows per thread, their loads in flight together.
constexpr int PAD_ROWS = 4;
__global__ void fft_pad_kernel(const void* img, int dtype, int H, int W, int pitch, const int* lohi, int R,
                               float* pad, int Wp) {
    const int X = blockIdx.x * blockDim.x + threadIdx.x;
    if (X >= W + 2 * R) return;
    const int lo = dtype == DTYPE_U16_STRETCH ? lohi[0] : 0, hi = dtype == DTYPE_U16_STRETCH ? lohi[1] : 0;
    const float rcp = stretch_rcp(lo, hi);
    const int x = refl(X - R, W), rows = H + 2 * R;
    for (int Y0 = PAD_ROWS * blockIdx.y; Y0 < rows; Y0 += PAD_ROWS * gridDim.y) {
        unsigned v[PAD_ROWS];
#pragma unroll
        for (int u = 0; u < PAD_ROWS; ++u) v[u] = load_raw(img, dtype, pitch, refl(min(Y0 + u, rows - 1) - R, H), x);
#pragma unroll
        for (int u = 0; u < PAD_ROWS; ++u)
            if (Y0 + u < rows) pad[(size_t)(Y0 + u) * Wp + X] = raw_to_px(v[u], dtype, lo, hi, rcp);
    }
}

// spectra of all levels: specs[i] = spec * gy[i][ky] * gx[i][kx]
__global__ void fft_levels_kernel(const cufftComplex* __restrict__ spec, const float* __restrict__ gx,
                                  const float* __restrict__ gy, int K, int Hp, int Wc, cufftComplex* specs) {
    const int kx = blockIdx.x * blockDim.x + threadIdx.x;
    if (kx >= Wc) return;
    const size_t n_spec = (size_t)Hp * Wc;
    for (int ky = blockIdx.y; ky < Hp; ky += gridDim.y) {
        const size_t o = (size_t)ky * Wc + kx;
        const cufftComplex s = spec[o];
        for (int i = 0; i < K; ++i) {
            const float g = __fmul_rn(gy[(size_t)i * Hp + ky], gx[(size_t)i * Wc + kx]);
            specs[(size_t)i * n_spec + o] = make_float2(__fmul_rn(s.x, g), __fmul_rn(s.y, g));
        }
    }
}

// DoG, 3x3x3 maximum and threshold from the level planes.  Neighbours outside
// the frame or the ladder do not count (-inf); ties keep the voxel (it equals its
// maximum filter); strict threshold D > thr.  mode MODE_CANDIDATES: compaction
// into blobs; MODE_DUMP: writes D.
//
// A warp takes 30 columns (lanes 1 .. 30; 0 and 31 are neighbours) by FT_ROWS
// rows and walks the planes: a level costs FT_ROWS + 2 loads per lane, the 3x3
// maximum three rows at a time and two shuffles, and a plane is settled when the
// next one's maxima exist.  (One thread per pixel with nine neighbours of both
// levels loaded for every plane took 42 us for 6 levels of 1024 x 1024; this
// takes 12.3.)  c > 0 and rounding is monotonic, so the maximum of the scaled
// differences is the scaled maximum.
constexpr int FT_ROWS = 4, FT_WARPS = 8;
template <int MODE>
__global__ void __launch_bounds__(32 * FT_WARPS) fft_test_kernel(const float* __restrict__ planes, int Hp, int Wp,
                                                                 int R, int H, int W, int P,
                                                                 const float* __restrict__ c, float thr,
                                                                 dog_blob* blobs, int cap, int* count, float* dump,
                                                                 int* status) {
    const int lane = threadIdx.x & 31;
    const int x = blockIdx.x * 30 + lane - 1;
    const int y0 = (blockIdx.y * FT_WARPS + (threadIdx.x >> 5)) * FT_ROWS;
    if (y0 >= H) return;
    const size_t plane = (size_t)Hp * Wp;
    const float NEG = -INFINITY;
    const bool col = x >= 0 && x < W, own = col && lane >= 1 && lane <= 30;
    // rows y0 - 1 .. y0 + FT_ROWS of the grid (clamped to the frame; masked below)
    const float* base = planes + (size_t)R * Wp + R + min(max(x, 0), W - 1);
    auto row = [&](int k) { return (size_t)min(max(y0 - 1 + k, 0), H - 1) * Wp; };
    float La[FT_ROWS + 2];
#pragma unroll
    for (int k = 0; k < FT_ROWS + 2; ++k) La[k] = base[row(k)];
    float m1[FT_ROWS], m2[FT_ROWS], e1[FT_ROWS];   // maxima of planes l-1, l-2; differences of plane l-1
#pragma unroll
    for (int t = 0; t < FT_ROWS; ++t) m1[t] = m2[t] = e1[t] = NEG;
    float cp = 1.0f;
    for (int l = 0; l <= P; ++l) {
        float m0[FT_ROWS], e0[FT_ROWS];
        float cl = 1.0f;
        if (l < P) {
            base += plane;
            cl = __ldg(c + l);
            float e[FT_ROWS + 2];
#pragma unroll
            for (int k = 0; k < FT_ROWS + 2; ++k) {
                const float b = base[row(k)];
                e[k] = col && y0 - 1 + k >= 0 && y0 - 1 + k < H ? __fsub_rn(La[k], b) : NEG;
                La[k] = b;
            }
#pragma unroll
            for (int t = 0; t < FT_ROWS; ++t) {
                e0[t] = e[t + 1];
                if (MODE == MODE_DUMP) {
                    if (own && y0 + t < H) dump[((size_t)l * H + y0 + t) * W + x] = __fmul_rn(cl, e0[t]);
                } else {
                    const float v = fmaxf(e[t], fmaxf(e[t + 1], e[t + 2]));
                    const float vl = __shfl_up_sync(0xffffffffu, v, 1), vr = __shfl_down_sync(0xffffffffu, v, 1);
                    m0[t] = __fmul_rn(cl, fmaxf(v, fmaxf(vl, vr)));
                }
            }
        } else {
#pragma unroll
            for (int t = 0; t < FT_ROWS; ++t) m0[t] = e0[t] = NEG;
        }
        if (MODE == MODE_DUMP) continue;
#pragma unroll
        for (int t = 0; t < FT_ROWS; ++t) {
            const float d = __fmul_rn(cp, e1[t]);
            if (own && y0 + t < H && d > thr && d >= fmaxf(m0[t], fmaxf(m1[t], m2[t]))) {
                const int idx = atomicAdd(count, 1);
                if (idx < cap) {
                    dog_blob b;
                    b.x = x; b.y = y0 + t; b.level = l - 1; b.sigma = c[P + l - 1]; b.response = d;
                    blobs[idx] = b;
                } else {
                    atomicCAS(status, 0, (int)DOG_ERR_CAPACITY);
                }
            }
            m2[t] = m1[t];
            m1[t] = m0[t];
            e1[t] = e0[t];
        }
        cp = cl;
    }
}

// The scale space of one frame on the FFT grid (planes), then the test.
int fft_run(FftWS* f, const void* img, int dtype, int H, int W, int pitch, const int* lohi, int P,
            const float* c, float thr, int mode, dog_blob* blobs, int cap, int* count, float* dump, int* status,
            cudaStream_t s) {
    if (H + 2 * f->R > f->Hp || W + 2 * f->R > f->Wp) return DOG_ERR_INVALID;
    const int Wc = f->Wp / 2 + 1;
    if ((H < f->last_h || W < f->last_w) &&   // cells a larger frame padded: back to zero
        cudaMemsetAsync(f->pad, 0, sizeof(float) * (size_t)f->Hp * f->Wp, s) != cudaSuccess)
        return DOG_ERR_CUDA;
    f->last_h = H;
    f->last_w = W;
    const int gy_pad = (H + 2 * f->R + PAD_ROWS - 1) / PAD_ROWS;   // (below 65535: frames have at most 65535 rows)
    fft_pad_kernel<<<dim3((W + 2 * f->R + 255) / 256, gy_pad), 256, 0, s>>>(img, dtype, H, W, pitch, lohi, f->R,
                                                                           f->pad, f->Wp);
    if (cudaGetLastError() != cudaSuccess) return DOG_ERR_CUDA;
    if (cufftSetStream(f->fwd, s) != CUFFT_SUCCESS || cufftSetStream(f->inv, s) != CUFFT_SUCCESS) return DOG_ERR_CUDA;
    if (cufftExecR2C(f->fwd, f->pad, f->spec) != CUFFT_SUCCESS) return DOG_ERR_CUDA;
    fft_levels_kernel<<<dim3((Wc + 255) / 256, f->Hp < 65535 ? f->Hp : 65535), 256, 0, s>>>(f->spec, f->gx, f->gy,
                                                                                         f->K, f->Hp, Wc, f->specs);
    if (cudaGetLastError() != cudaSuccess) return DOG_ERR_CUDA;
    if (cufftExecC2R(f->inv, f->specs, f->planes) != CUFFT_SUCCESS) return DOG_ERR_CUDA;
    if (mode == MODE_CANDIDATES && cudaMemsetAsync(count, 0, sizeof(int), s) != cudaSuccess) return DOG_ERR_CUDA;
    const dim3 grid((W + 29) / 30, (H + FT_ROWS * FT_WARPS - 1) / (FT_ROWS * FT_WARPS));
    if (mode == MODE_CANDIDATES)
        fft_test_kernel<MODE_CANDIDATES><<<grid, 32 * FT_WARPS, 0, s>>>(f->planes, f->Hp, f->Wp, f->R, H, W, P, c, thr,
                                                                        blobs, cap, count, dump, status);
    else
        fft_test_kernel<MODE_DUMP><<<grid, 32 * FT_WARPS, 0, s>>>(f->planes, f->Hp, f->Wp, f->R, H, W, P, c, thr, blobs,
                                                                  cap, count, dump, status);
    return cudaGetLastError() == cudaSuccess ? DOG_OK : DOG_ERR_CUDA;
}

}  // namespace dogk

// Contrast stretch of 12-bit frames (Sec. 4: the optional first step maps a
// frame to [0, 1] with 0.35% saturation; Table 2 shows it dominating the
// paper's CPU preprocessing).
//
// Reading: with the frame's n counts sorted ascending and k = floor(sat/2 n),
// the count at rank k maps to 0, the count at rank n-1-k maps to 1, and the
// map (c - lo) / (hi - lo) is clipped to [0, 1]; counts above 4095 count as
// 4095.  On the GPU the order statistics come from a 4096-bin histogram per
// frame (shared-memory counts, one global atomic per nonzero bin and CTA) and
// a scan of it by the frame's last CTA; the map itself is applied where the
// detection kernels ingest the frame (stretch_px) or by stretch_apply_kernel.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "dog_internal.cuh"
#include "dog_device.cuh"

namespace dogk {

constexpr int HIST_THREADS = 512, HIST_WARPS = HIST_THREADS / 32;
constexpr int BINS_EACH = STRETCH_BINS / HIST_THREADS;   // bins of a thread in the limits scan

constexpr int UNIT = 512;   // counts of a row that a warp takes at a time: two loads of eight per lane

// Histogram of frame blockIdx.y by units of its rows, the warps of all its CTAs in
// turn; then the limits by
// the CTA that finishes last: the counts at ranks k and n-1-k (k = floor(sat/2 n),
// at most (n-1)/2) are the bins v with #(c < v) <= rank < #(c <= v).
// frames == nullptr: the single frame (img, H, W, pitch).  hist: STRETCH_BINS
// words per frame, zeroed by the caller; the last one counts the finished CTAs
// (the last bin is what the others leave of the n pixels).  lohi[2f] = lo,
// lohi[2f+1] = hi.  The additions to the frame's bins bound it (1024 x 1280, with
// the limits): one CTA of 512 threads per SM takes 7.8 us, two of 256 take 11.6;
// one count per load in 6 us and the limits as a launch of their own, 3 us and
// the gap between, came before.
__global__ void __launch_bounds__(HIST_THREADS) stretch_limits_kernel(const dog_frame* frames, const uint16_t* img,
                                                                      int H, int W, int pitch, double sat, int* hist,
                                                                      int* lohi) {
    __shared__ int sh[STRETCH_BINS];
    __shared__ int wsum[HIST_WARPS];
    __shared__ bool last;
    const int f = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (frames) {
        const dog_frame fr = frames[f];
        if (fr.dtype != DOG_DTYPE_U16) return;   // only 12-bit frames are stretched
        img = static_cast<const uint16_t*>(fr.ptr);
        H = fr.h;
        W = fr.w;
        pitch = fr.pitch;
    }
    for (int q = tid; q < STRETCH_BINS; q += HIST_THREADS) sh[q] = 0;
    __syncthreads();
    auto add = [&](unsigned v) { atomicAdd(&sh[min(v, (unsigned)STRETCH_BINS - 1)], 1); };
    const int units = max(1, (W + UNIT - 1) / UNIT);   // of a row
    const long long all = (long long)H * units;
    for (long long i = blockIdx.x * HIST_WARPS + warp; i < all; i += gridDim.x * HIST_WARPS) {
        const int y = (int)(i / units), u = (int)(i - (long long)y * units);
        const uint16_t* row = img + (size_t)y * pitch;
        const int head = min(W, (int)((16 - (reinterpret_cast<size_t>(row) & 15)) & 15) / 2), n8 = (W - head) / 8;
        const uint4* row8 = reinterpret_cast<const uint4*>(row + head);
        const int x = u * (UNIT / 8) + lane;
        uint4 v[2];
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (x + 32 * k < n8) v[k] = __ldg(row8 + x + 32 * k);
        if (u == 0) {
            if (lane < head) add(__ldg(row + lane));
            for (int t = head + 8 * n8 + lane; t < W; t += 32) add(__ldg(row + t));
        }
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (x + 32 * k < n8) {
                add(v[k].x & 0xffffu); add(v[k].x >> 16); add(v[k].y & 0xffffu); add(v[k].y >> 16);
                add(v[k].z & 0xffffu); add(v[k].z >> 16); add(v[k].w & 0xffffu); add(v[k].w >> 16);
            }
    }
    __syncthreads();
    int* out = hist + (size_t)f * STRETCH_BINS;
    for (int q = tid; q < STRETCH_BINS - 1; q += HIST_THREADS)
        if (sh[q]) atomicAdd(&out[q], sh[q]);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&out[STRETCH_BINS - 1], 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const long long n = (long long)H * W;
    long long k = (long long)floor(sat * 0.5 * (double)n);
    if (k > (n - 1) / 2) k = (n - 1) / 2;
    const long long r_lo = k, r_hi = n - 1 - k;
    int c[BINS_EACH];
    int tsum = 0;
    const int* mine = out + BINS_EACH * tid;
    if ((reinterpret_cast<size_t>(out) & 15) == 0) {
#pragma unroll
        for (int u = 0; u < BINS_EACH; u += 4) {
            const int4 b = __ldcg(reinterpret_cast<const int4*>(mine + u));
            c[u] = b.x; c[u + 1] = b.y; c[u + 2] = b.z; c[u + 3] = b.w;
        }
    } else {   // the scratch is the caller's, of any alignment of an int
#pragma unroll
        for (int u = 0; u < BINS_EACH; ++u) c[u] = __ldcg(mine + u);
    }
    if (tid == HIST_THREADS - 1) c[BINS_EACH - 1] = 0;
#pragma unroll
    for (int u = 0; u < BINS_EACH; ++u) tsum += c[u];
    // block exclusive scan of the per-thread sums
    int incl = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    long long below = incl - tsum;   // #(c < BINS_EACH tid)
    for (int w = 0; w < warp; ++w) below += wsum[w];
    if (tid == HIST_THREADS - 1) c[BINS_EACH - 1] = (int)(n - below - tsum);
#pragma unroll
    for (int u = 0; u < BINS_EACH; ++u) {
        const long long upto = below + c[u];   // #(c <= v)
        const int v = BINS_EACH * tid + u;
        if (below <= r_lo && r_lo < upto) lohi[2 * f] = v;
        if (below <= r_hi && r_hi < upto) lohi[2 * f + 1] = v;
        below = upto;
    }
}

// The stretched frame (FP32, [0, 1]) of one 12-bit frame with limits lohi.
// Row blockIdx.y (grid-strided); each thread maps 4 consecutive pixels, with
// one 8-byte load and one 16-byte store when both rows allow it.
__global__ void __launch_bounds__(256) stretch_apply_kernel(const uint16_t* img, int H, int W, int pitch,
                                                            const int* lohi, float* out, int out_pitch) {
    const int lo = lohi[0], hi = lohi[1];
    const float rcp = stretch_rcp(lo, hi);
    for (int y = blockIdx.y; y < H; y += gridDim.y) {
        const uint16_t* src = img + (size_t)y * pitch;
        float* dst = out + (size_t)y * out_pitch;
        const bool vec = ((reinterpret_cast<size_t>(src) & 7) == 0) && ((reinterpret_cast<size_t>(dst) & 15) == 0);
        for (int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x); x < W; x += 4 * gridDim.x * blockDim.x) {
            if (vec && x + 4 <= W) {
                const uint2 v = __ldg(reinterpret_cast<const uint2*>(src + x));
                *reinterpret_cast<float4*>(dst + x) =
                    make_float4(stretch_px(v.x & 0xffffu, lo, hi, rcp), stretch_px(v.x >> 16, lo, hi, rcp),
                                stretch_px(v.y & 0xffffu, lo, hi, rcp), stretch_px(v.y >> 16, lo, hi, rcp));
            } else {
                for (int u = x; u < x + 4 && u < W; ++u) dst[u] = stretch_px(__ldg(src + u), lo, hi, rcp);
            }
        }
    }
}

cudaError_t launch_stretch_limits(const dog_frame* frames, int n, const uint16_t* img, int H, int W, int pitch,
                                  double sat, int num_sms, int* hist, int* lohi, cudaStream_t s) {
    if (n < 1 || n > 65535) return cudaErrorInvalidValue;   // frames index the grid's y dimension
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(int) * STRETCH_BINS * (size_t)n, s);
    if (e != cudaSuccess) return e;
    // about one CTA per SM over the whole call; a frame's warps split its rows' units
    int per = (num_sms + n - 1) / n;
    if (!frames) {
        const long long all = (long long)H * ((W + UNIT - 1) / UNIT);
        per = (int)std::min<long long>(per, (all + HIST_WARPS - 1) / HIST_WARPS);
    }
    stretch_limits_kernel<<<dim3(per, n), HIST_THREADS, 0, s>>>(frames, img, H, W, pitch, sat, hist, lohi);
    return cudaGetLastError();
}

cudaError_t launch_stretch_apply(const uint16_t* img, int H, int W, int pitch, const int* lohi, float* out,
                                 int out_pitch, int num_sms, cudaStream_t s) {
    const int gx = (W + 4 * 256 - 1) / (4 * 256);
    int gy = (8 * num_sms + gx - 1) / gx;
    if (gy > H) gy = H;
    if (gy > 65535) gy = 65535;
    stretch_apply_kernel<<<dim3(gx, gy), 256, 0, s>>>(img, H, W, pitch, lohi, out, out_pitch);
    return cudaGetLastError();
}

}  // namespace dogk

using namespace dogk;

extern "C" int dog_stretch_limits(const uint16_t* d_img, int32_t img_h, int32_t img_w, int32_t pitch, double sat,
                                  int32_t* d_hist, int32_t* d_lohi, void* stream) {
    if (!d_img || !d_hist || !d_lohi || img_h < 1 || img_w < 1 || pitch < img_w) return DOG_ERR_INVALID;
    if (!(sat >= 0.0 && sat < 1.0)) return DOG_ERR_INVALID;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return DOG_ERR_CUDA;
    return launch_stretch_limits(nullptr, 1, d_img, img_h, img_w, pitch, sat, sms, d_hist, d_lohi,
                                 static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? DOG_OK
               : DOG_ERR_CUDA;
}

extern "C" int dog_stretch(const uint16_t* d_img, int32_t img_h, int32_t img_w, int32_t pitch,
                           const int32_t* d_lohi, float* d_out, int32_t out_pitch, void* stream) {
    if (!d_img || !d_lohi || !d_out || img_h < 1 || img_w < 1 || pitch < img_w || out_pitch < img_w)
        return DOG_ERR_INVALID;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return DOG_ERR_CUDA;
    return launch_stretch_apply(d_img, img_h, img_w, pitch, d_lohi, d_out, out_pitch, sms,
                                static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? DOG_OK
               : DOG_ERR_CUDA;
}

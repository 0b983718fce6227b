// Synthetic sphere frames on the GPU (Sec. 5 evaluates the detector on
// frames of 100 rendered spheres with Poisson and Gaussian noise; the paper
// names no shading model).
//
// Reading: each sphere is an optically thin fluorescent droplet, so a pixel's
// brightness is proportional to the chord length through the sphere,
// sqrt(1 - d^2 / R^2) at distance d from the centre, averaged over ss x ss
// sub-pixel samples (pixel centres at integer coordinates); the frame is a
// background plus the spheres' contributions in table order, every step an
// explicitly rounded single-precision operation.  Counts are
//   floor(lambda + sqrt(lambda) z1 + read_noise z2 + 1/2) clipped to [0, 4095],
//   lambda = gain * intensity, in double,
// with z1, z2 sums of twelve uniforms minus 6; the uniforms are the top 24
// bits of Philox4x32-10 blocks (Salmon et al., SC'11), counter (pixel index
// low, high, draw, 0), key (seed low, high), three blocks per normal.
//
// A CTA renders a 32 x 32 tile: it first lists, in table order, the spheres
// whose disc (plus one pixel) meets the tile; spheres left out contribute
// exactly zero to every sample of the tile, so the sums are unchanged (see
// beside).  A warp
// then takes four blocks of 16 x 2 pixels and skips the listed spheres that miss
// its block.  Frames of few tiles give a tile's blocks to two or four CTAs, which
// list the same spheres each.
//
// What bounds it: integer multiplies of the generator (six Philox blocks a
// pixel).  The double-precision pipe (two lanes a cycle and SM here) was the
// bound before: 24 additions and products per normal and the count itself, 1476
// us for 8 frames of 1000 x 1000 with 100 spheres.  The uniforms are multiples of
// 2^-24, so a normal's sum is an integer; the count is decided in single
// precision, with the double-precision formula only for the pixels that come
// within the error bound of a rounding edge (below 1%): 226 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cfloat>

#include "dog.h"

namespace {

constexpr int RT = 32;                 // tile edge
constexpr int RTHREADS = 256;
constexpr int MAX_SPHERES = 8192;      // shared-memory list of one tile

__device__ __forceinline__ void philox4x32_10(uint32_t (&c)[4], uint32_t k0, uint32_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c[0], p1 = (uint64_t)0xCD9E8D57u * c[2];
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c[1] ^ k0, n2 = (uint32_t)(p0 >> 32) ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = (uint32_t)p1;
        c[2] = n2;
        c[3] = (uint32_t)p0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

// Twelve uniforms of 24 bits, summed as integers: the normal is sum 2^-24 - 6,
// exact in double.
__device__ __forceinline__ uint32_t sum12(unsigned long long pix, uint32_t draw0, uint32_t k0, uint32_t k1) {
    uint32_t s = 0;
#pragma unroll
    for (uint32_t b = 0; b < 3; ++b) {
        uint32_t c[4] = {(uint32_t)pix, (uint32_t)(pix >> 32), draw0 + b, 0u};
        philox4x32_10(c, k0, k1);
#pragma unroll
        for (int q = 0; q < 4; ++q) s += c[q] >> 8;
    }
    return s;
}

// The sphere (cx, cy, R, A) contributes exactly zero to every sample of the pixels
// x0 .. x1, y0 .. y1: its disc and a pixel around it are beside them.  R enters as
// R^2 only, so its sign does not count.  Of larger spheres the rounding of d^2 /
// R^2 could let a sample outside the disc through (R = 5e6: 1 - d^2 / R^2 is 4e-7
// a pixel outside, with an error of up to 3e-7), and an amplitude that is not
// finite makes even a zero count: those are never left out.
__device__ __forceinline__ bool beside(const float4& q, float x0, float x1, float y0, float y1) {
    const float m = fabsf(q.z) + 1.0f;
    const bool meets = q.x + m >= x0 - 0.5f && q.x - m <= x1 + 0.5f && q.y + m >= y0 - 0.5f && q.y - m <= y1 + 0.5f;
    return !meets && m < 1.0e6f && fabsf(q.w) < INFINITY;
}

// The count of one pixel as defined, in double.
__device__ __noinline__ uint16_t count_exact(double gain, float I, double read_noise, uint32_t s1, uint32_t s2) {
    const double z1 = (double)s1 * (1.0 / 16777216.0) - 6.0, z2 = (double)s2 * (1.0 / 16777216.0) - 6.0;
    const double lam = __dmul_rn(gain, (double)I);
    const double sl = __dsqrt_rn(lam > 0.0 ? lam : 0.0);
    double v = floor(__dadd_rn(__dadd_rn(__dadd_rn(lam, __dmul_rn(sl, z1)), __dmul_rn(read_noise, z2)), 0.5));
    v = v < 0.0 ? 0.0 : (v > 4095.0 ? 4095.0 : v);
    return (uint16_t)v;
}

__global__ void __launch_bounds__(RTHREADS) render_spheres_kernel(const float4* __restrict__ sph, int S, int H,
                                                                  int W, int ss, float bg, double gain,
                                                                  double read_noise, uint32_t k0, uint32_t k1,
                                                                  float* inten, uint16_t* counts, int pitch) {
    __shared__ int list[MAX_SPHERES];
    __shared__ int wsum[RTHREADS / 32];
    __shared__ int n_list;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x0 = blockIdx.x * RT, y0 = blockIdx.y * RT;
    if (tid == 0) n_list = 0;
    __syncthreads();
    // spheres meeting the tile, in table order (chunks of RTHREADS, block scan)
    for (int base = 0; base < S; base += RTHREADS) {
        const int s = base + tid;
        bool keep = false;
        if (s < S)
            keep = !beside(__ldg(sph + s), (float)x0, (float)(x0 + RT - 1), (float)y0, (float)(y0 + RT - 1));
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) wsum[warp] = __popc(mask);
        __syncthreads();
        int at = n_list, total = 0;
        for (int w = 0; w < RTHREADS / 32; ++w) {
            at += (w < warp) ? wsum[w] : 0;
            total += wsum[w];
        }
        if (keep) list[at + __popc(mask & ((1u << lane) - 1u))] = s;
        __syncthreads();
        if (tid == 0) n_list += total;
        __syncthreads();
    }
    const int n = n_list;
    const float inv_n = 1.0f / (float)(ss * ss), half_ss = 0.5f / (float)ss;   // exact: ss is a power of two
    // (a gain below the normal range of single precision has lost digits: NaN, so
    // that no count is decided in single precision)
    const float gain_f = fabs(gain) < (double)FLT_MIN && gain != 0.0 ? NAN : (float)gain, rn_f = (float)read_noise;
#pragma unroll 1
    for (int blk = blockIdx.z; blk < 4; blk += gridDim.z) {
        // block of 16 x 2 pixels: warp rows 4 w .. 4 w + 3, two blocks side by side
        const int bx = x0 + (blk & 1) * 16, by = y0 + 4 * warp + (blk >> 1) * 2;
        if (bx >= W || by >= H) continue;
        const int x = bx + (lane & 15), y = by + (lane >> 4);
        float I = bg;
        for (int t = 0; t < n; ++t) {
            const float4 q = __ldg(sph + list[t]);
            if (beside(q, (float)bx, (float)(bx + 15), (float)by, (float)(by + 1))) continue;
            const float inv_r2 = __fdiv_rn(1.0f, __fmul_rn(q.z, q.z));
            float acc = 0.0f;
            for (int j = 0; j < ss; ++j) {
                const float v = __fadd_rn((float)y, __fsub_rn(__fmul_rn((float)(2 * j + 1), half_ss), 0.5f));
                const float dy = __fsub_rn(v, q.y);
                const float dy2 = __fmul_rn(dy, dy);
                for (int i = 0; i < ss; ++i) {
                    const float u = __fadd_rn((float)x, __fsub_rn(__fmul_rn((float)(2 * i + 1), half_ss), 0.5f));
                    const float dx = __fsub_rn(u, q.x);
                    const float qq = __fsub_rn(1.0f, __fmul_rn(__fadd_rn(__fmul_rn(dx, dx), dy2), inv_r2));
                    if (qq > 0.0f) acc = __fadd_rn(acc, __fsqrt_rn(qq));
                }
            }
            I = __fadd_rn(I, __fmul_rn(q.w, __fmul_rn(acc, inv_n)));
        }
        if (x >= W || y >= H) continue;
        if (inten) inten[(size_t)y * W + x] = I;
        const unsigned long long pix = (unsigned long long)y * (unsigned long long)W + (unsigned long long)x;
        const uint32_t s1 = sum12(pix, 0u, k0, k1), s2 = sum12(pix, 3u, k0, k1);
        // single precision: s1 - 6 2^24 is below 2^27, so z is off by 2^-23 of its
        // size; every term of v below by a few 2^-24 of its size; 1e-6 covers them
        const float z1 = (float)((int)s1 - 6 * 16777216) * (1.0f / 16777216.0f);
        const float z2 = (float)((int)s2 - 6 * 16777216) * (1.0f / 16777216.0f);
        const float lam = gain_f * I, shot = sqrtf(fmaxf(lam, 0.0f)) * z1, read = rn_f * z2;
        const float v = lam + shot + read + 0.5f, off = 1e-6f * (fabsf(lam) + fabsf(shot) + fabsf(read) + 1.0f);
        const float fl = floorf(v);
        uint16_t c;
        if (v - fl > off && fl + 1.0f - v > off) c = (uint16_t)fminf(fmaxf(fl, 0.0f), 4095.0f);
        else c = count_exact(gain, I, read_noise, s1, s2);   // (not-a-numbers too)
        counts[(size_t)y * pitch + x] = c;
    }
}

}  // namespace

extern "C" int dog_render_spheres(const float* d_spheres, int32_t n_spheres, int32_t img_h, int32_t img_w,
                                  int32_t ss, float background, double gain, double read_noise, uint64_t seed,
                                  float* d_intensity, uint16_t* d_counts, int32_t pitch, void* stream) {
    if ((n_spheres > 0 && !d_spheres) || n_spheres < 0 || !d_counts || img_h < 1 || img_w < 1 || pitch < img_w)
        return DOG_ERR_INVALID;
    if (!(ss == 1 || ss == 2 || ss == 4 || ss == 8)) return DOG_ERR_INVALID;
    if (n_spheres > MAX_SPHERES) return DOG_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(d_spheres) & 15) != 0) return DOG_ERR_INVALID;
    dim3 grid((img_w + RT - 1) / RT, (img_h + RT - 1) / RT);
    if (grid.y > 65535) return DOG_ERR_UNSUPPORTED;
    // CTAs per tile: up to 2560 in all, two and a half times what is resident.  Four
    // blocks to a CTA leave the SMs idle on fewer tiles (64 x 64 pixels 51 us, with
    // four CTAs a tile 16; 512 x 512 19.3, 12.1; 1000 x 1000 with two 30.8, 27.2);
    // on more the lists cost more than that (2000 x 2000 74.9, with two 81.0)
    const long long tiles = (long long)grid.x * grid.y;
    grid.z = tiles <= 640 ? 4 : tiles <= 1280 ? 2 : 1;
    render_spheres_kernel<<<grid, RTHREADS, 0, static_cast<cudaStream_t>(stream)>>>(
        reinterpret_cast<const float4*>(d_spheres), n_spheres, img_h, img_w, ss, background, gain, read_noise,
        (uint32_t)seed, (uint32_t)(seed >> 32), d_intensity, d_counts, pitch);
    return cudaGetLastError() == cudaSuccess ? DOG_OK : DOG_ERR_CUDA;
}

// Fused DoG detector kernel for sm_103a: the kernel forms, templated on the
// number of warps, the mode and the source of tiles (dog_fused.cu and
// dog_fused_w10/w8/w4/w3/w2.cu instantiate them).
//
// Method (arXiv 2010.08486): scale space L_i = g(sigma_i) * I (Sec. 3), DoG
// D_i = c_i (L_i - L_{i+1}) (Eq. 2-3), voxels equal to their 3x3x3 maximum
// and above the threshold (Sec. 4, Sec. 4.1).
//
// Design.  A CTA owns a strip of TX = 32 output columns and walks down a band
// of rows in blocks of 8 NW rows, one chunk of 8 rows per warp, so every input
// pixel of the strip is read once from global memory for all K scales.  Within
// a block the levels are taken two at a time (a pair), all warps on the same
// pair: in interval p a warp runs
//   1. the maximum test of the two planes formed in the interval before,
//   2. the horizontal pass of pair p + 1 for its 8 rows, into shared memory,
//   3. the vertical pass of pair p for its 8 rows, into registers,
//   4. the two differences the pair completes, in registers; it publishes the
//      last two rows of each for the warp below,
// and one barrier ends the interval.  The rows above a block that the vertical
// pass needs are kept per pair in a ring of chunks (2r rows; the horizontal
// pass is never repeated inside a band); the block's own chunks live in a
// double buffer shared by all pairs.
//
// What bounds it: FP32 multiply-adds (2 sum(2r+1) per pixel).  The two levels
// of a pair are the two lanes of packed FMAs, which halves the instructions and
// shares the input loads of the horizontal pass.  All warps work on one pair at
// a time so that the tap addresses are uniform and the taps come from the
// constant bank (the kernel's parameters) as uniform operands: with taps read
// from shared memory into registers the same inner loop takes 174 cycles per 64
// packed FMAs and scheduler instead of 135 (128 is the pipe's limit), because
// three register operands of 64 bits leave no register bandwidth for the loads
// that fill the windows.  It also gives every warp the same work, so nobody
// waits at the barrier, and the L rows never go through shared memory.
//
// Measured (96 frames of 1024 x 1024, 12-bit, one batched launch): 25 levels to
// sigma 7.9 9.87 -> 8.24 ms, 12 levels 1.25^k 9.18 -> 5.65 ms, 6 levels to sigma
// 10.5 6.69 -> 3.52 ms (12 warps), 14 levels to sigma 12.3 10.56 -> 8.25 ms (10
// warps), against the form before (levels on fixed producer warps, scalar FMAs,
// taps and L rows through shared memory).  A block is 8 NW rows, so tiles that fill
// little of one gain least: 25 levels on batched frames of 32 rows or fewer, or of
// 97, take 5 to 14% longer than the form before (with 8 warps as long as with 12);
// other ladders are faster there too.
//
// Both passes are register-blocked 1-D correlations: 8 outputs per lane, taps
// in blocks of 8 against a two-window register file whose halves swap roles
// each block, so one short loop serves every radius.  The taps of both levels
// sit in the wider level's window, zero-padded to 8 ceil((2r+1)/8); they are
// summed in ascending order with FMA from zero, so the padding never changes a
// (finite) value and the resolve kernel (dog_resolve.cu), which repeats the
// order on the real taps only, reproduces any response bit for bit.
// Neighbours in the adjacent strip are not held here: in detection a candidate
// at a strip edge is queued and the resolve kernel recomputes the few responses
// it needs; the soft modes, which keep every local maximum (thousands at strip
// edges per frame), instead step 32-column strips by 30 so that lanes 0 and 31
// are only neighbours and every voxel a strip owns has its whole neighbourhood.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cfloat>

#include "dog_internal.cuh"
#include "dog_device.cuh"

namespace dogk {

// Where a tile's input pixels come from.
struct PixelSource {
    const void* img;
    int dtype, H, W, pitch;
    int st_lo, st_hi;
    float st_rcp;
    int x0;
};

struct TileCtx {
    const void* img;
    int dtype, H, W, pitch;
    int st_lo, st_hi;   // contrast-stretch limits (DTYPE_U16_STRETCH)
    float st_rcp;       // stretch_rcp(st_lo, st_hi)
    int frame;
    int x0, y0, y1;
    dog_blob* blobs;
    int* count;
};

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Shared scalars of one CTA (static shared memory: SMEM_RESERVE).
struct SmemSmall {
    float c[MAX_LEVELS];      // normalisation (soft modes: its size; sg has the sign)
    float sig[MAX_LEVELS];
    float gk[MAX_LEVELS];     // sum_b gH_b kappa_b(t_l)
    float gdk[MAX_LEVELS];    // sum_b gH_b dkappa_b/dt(t_l)
    int kb[MAX_LEVELS][2];    // nonzero soft-histogram bins of each plane
    float kw[MAX_LEVELS][2];
    float soft[DOG_MAX_NBINS];
    float dc[MAX_LEVELS];
    float dt[MAX_LEVELS];
    PixelSource px;           // the tile in work (load8 reads it here: fewer registers held)
    int tile;
    float sg[MAX_LEVELS];     // soft modes: the sign of c
    int flip;                 // soft modes: some c is negative
    int careful;              // a pixel of the tile is not finite (or huge): correlate_exact
};
static_assert(sizeof(SmemSmall) <= SMEM_RESERVE, "reserved next to the dynamic shared memory");

// Pixels beyond this magnitude take the careful path (their sums may overflow).
constexpr float HUGE_PX = 1e37f;

// ---------------------------------------------------------------------------
// Taps of a pair, four floats (two taps of two levels) at a time: from the
// kernel's parameters (constant bank), or from shared memory when the taps are
// device data (soft modes).
template <bool CT>
struct Taps {
    const FusedParams& p;
    const float4* sm;
    __device__ __forceinline__ float4 operator()(int q) const { return CT ? p.taps[q] : sm[q]; }
};

// acc[k] += (w_lo[u], w_hi[u]) * X[k + u], u = 0..7: both levels on the same
// input (horizontal pass) or each on its own (vertical pass).
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 both(float2 x) { return x; }

template <class T, bool CT>
__device__ __forceinline__ void fma_block(float2 (&acc)[8], const T (&A)[8], const T (&B)[8], const Taps<CT>& tap,
                                          int q) {
#pragma unroll
    for (int u2 = 0; u2 < 4; ++u2) {
        const float4 w4 = tap(q + u2);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int u = 2 * u2 + v;
            const float2 w = v ? make_float2(w4.z, w4.w) : make_float2(w4.x, w4.y);
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = __ffma2_rn(w, both((k + u < 8) ? A[k + u] : B[k + u - 8]), acc[k]);
        }
    }
}

// The single last tap of a window whose 2r + 1 taps are one more than a
// multiple of 8 (the rest of its padded block is zeros).
template <class T, bool CT>
__device__ __forceinline__ void fma_tail(float2 (&acc)[8], const T (&Y)[8], const Taps<CT>& tap, int q) {
    const float4 w4 = tap(q);
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = __ffma2_rn(make_float2(w4.x, w4.y), both(Y[k]), acc[k]);
}

// out[k] = sum_u w[u] X[k + u] over nb blocks of 8 taps (and the tail);
// load(A) fetches the next 8 inputs of the window.
template <class T, bool CT, class Load>
__device__ __forceinline__ void correlate(float2 (&acc)[8], Load load, const Taps<CT>& tap, int q, int nb, bool tail) {
    T A[8], B[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = make_float2(0.0f, 0.0f);
    load(A);
    for (;;) {
        load(B);
        fma_block(acc, A, B, tap, q);
        q += 4;
        if (--nb == 0) {
            if (tail) fma_tail(acc, B, tap, q);
            break;
        }
        load(A);
        fma_block(acc, B, A, tap, q);
        q += 4;
        if (--nb == 0) {
            if (tail) fma_tail(acc, A, tap, q);
            break;
        }
    }
}

// The same sums over each level's real taps only, for tiles with non-finite (or
// huge) pixels: a zero tap of the padded windows would turn an infinity outside
// the level's own window into a NaN.  For finite inputs the zero taps add
// nothing, so both forms give the same bits.  The pair's window has 2 r + 1 taps,
// of which the first level has those from d to 2 r - d.  Blocks of taps that both
// levels have are taken as above; the others tap by tap.  (A loop over taps with
// loads of its own per level made the detection of a 1024 x 1024 frame with one
// such pixel take 680 us; this 240, and without such pixels 165.)
__device__ __forceinline__ float second(float x) { return x; }
__device__ __forceinline__ float second(float2 x) { return x.y; }

template <class T, bool CT>
__device__ __forceinline__ void exact_block(float2 (&acc)[8], const T (&A)[8], const T (&B)[8], const Taps<CT>& tap,
                                            int q, int t0, int d, int last) {
    if (t0 >= d && t0 + 7 <= last - d) {
        fma_block(acc, A, B, tap, q);
        return;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float4 w4 = tap(q + (u >> 1));
        const float2 w = u & 1 ? make_float2(w4.z, w4.w) : make_float2(w4.x, w4.y);
        if (t0 + u >= d && t0 + u <= last - d) {
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k] = __ffma2_rn(w, both((k + u < 8) ? A[k + u] : B[k + u - 8]), acc[k]);
        } else if (t0 + u <= last) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                acc[k].y = __fmaf_rn(w.y, second((k + u < 8) ? A[k + u] : B[k + u - 8]), acc[k].y);
        }
    }
}

template <class T, bool CT, class Load>
__device__ __forceinline__ void correlate_exact(float2 (&acc)[8], Load load, const Taps<CT>& tap, int q, int nb,
                                                bool tail, int d, int last) {
    T A[8], B[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = make_float2(0.0f, 0.0f);
    load(A);
#pragma unroll 1
    for (int t = 0; t < 8 * nb; t += 8) {
        load(B);
        exact_block(acc, A, B, tap, q, t, d, last);
        q += 4;
#pragma unroll
        for (int k = 0; k < 8; ++k) A[k] = B[k];
    }
    if (tail) {   // tap 8 nb, the last one: both levels' if their windows are the same
        if (d == 0) {
            fma_tail(acc, A, tap, q);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) acc[k].y = __fmaf_rn(tap(q).y, second(A[k]), acc[k].y);
        }
    }
}

// ---------------------------------------------------------------------------
// Chunks: 8 rows of a pair's horizontal sums, CHUNK floats; a row is 64 floats,
// column x's two levels at 2x.  The row's sixteen 16-byte pieces 4g + j sit at
// 4g + (j ^ chunk_swz), so that the horizontal pass's stores (lane (rho, g)
// writes pieces 4g .. 4g+3 of row rho) touch every bank once per quarter-warp.
__device__ __forceinline__ int chunk_swz(int row, int g) { return (g >> 1) | ((row & 1) << 1); }
__device__ __forceinline__ int chunk_off(int row, int x) {   // float offset of column x in row `row`
    const int g = x >> 3, j = (x >> 1) & 3;
    return row * PAIR_STRIDE + 4 * (4 * g + (j ^ chunk_swz(row, g))) + 2 * (x & 1);
}

// Sums of the horizontal pass into a chunk.
__device__ __forceinline__ void store_sums(float* dst, int rho, int g, const float2 (&acc)[8]) {
    float4* d4 = reinterpret_cast<float4*>(dst + rho * PAIR_STRIDE + 16 * g);
    const int swz = chunk_swz(rho, g);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        d4[j ^ swz] = make_float4(acc[2 * j].x, acc[2 * j].y, acc[2 * j + 1].x, acc[2 * j + 1].y);
}

// The horizontal pass over real taps only, src as in hpass.  Out of line: inlined
// beside the usual path it changes that one's registers (one frame of 1024 x 1024
// 124 -> 140 us).
template <bool CT>
__device__ __noinline__ void hpass_exact(const FusedParams& p, const PairInfo& U, const float* sm, const float* src,
                                         float* dst) {
    const Taps<CT> tap{p, reinterpret_cast<const float4*>(sm + p.t_off)};
    const int lane = threadIdx.x & 31, rho = lane >> 2, g = lane & 3;
    float2 acc[8];
    correlate_exact<float>(acc, [&](float (&X)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) X[k] = src[k];
        src += 8;
    }, tap, U.tap, U.nb, U.tail != 0, U.lead, 2 * U.r);
    store_sums(dst, rho, g, acc);
}

// Horizontal pass of pair U for 8 rows: lane (rho, g) columns 8g .. 8g+7 of row
// rho; row: this lane's input row (column 0 is frame column x0 - R).
template <bool CT>
__device__ __forceinline__ void hpass(const PairInfo& U, const float* sm, const float* row, int R, float* dst,
                                      const Taps<CT>& tap, bool careful) {
    const int lane = threadIdx.x & 31, rho = lane >> 2, g = lane & 3;
    const float* src = row + (R - U.r) + 8 * g;
    if (careful) {
        hpass_exact<CT>(tap.p, U, sm, src, dst);
        return;
    }
    float2 acc[8];
    correlate<float>(acc, [&](float (&X)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) X[k] = src[k];
        src += 8;
    }, tap, U.tap, U.nb, U.tail != 0);
    store_sums(dst, rho, g, acc);
}

// Vertical pass of pair U for chunk w of the block: lane = column.  The window
// is chunks at[0] .. at[e] (float offsets in sm): at points into the pair's
// table of logical chunks (chunk_table).  A table, because address arithmetic
// with comparisons in the loop makes the compiler give up the uniform tap
// operands (215 cycles per tap block against 155).
template <bool CT>
__device__ __forceinline__ void vpass(const PairInfo& U, const float* sm, const int* at, const Taps<CT>& tap,
                                      bool careful, float2 (&acc)[8]) {
    const int lane = threadIdx.x & 31;
    const int off_e = chunk_off(0, lane), off_o = chunk_off(1, lane);
    auto load = [&](float2 (&X)[8]) {
        const float* c = sm + *at++;
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            X[k] = *reinterpret_cast<const float2*>(c + off_e + k * PAIR_STRIDE);
            X[k + 1] = *reinterpret_cast<const float2*>(c + off_o + k * PAIR_STRIDE);
        }
    };
    if (!careful) correlate<float2>(acc, load, tap, U.tap, U.nb, U.tail != 0);
    else correlate_exact<float2>(acc, load, tap, U.tap, U.nb, U.tail != 0, U.lead, 2 * U.r);
}

// n mod e without a division (n < 2^28, e <= 17; rcp = ceil(2^32 / e), 0 for e = 1).
__device__ __forceinline__ int ring_pos(const PairInfo& U, int n) {
    return U.rcp ? n - (int)__umulhi((unsigned)n, U.rcp) * U.e : 0;
}

// Offsets of a pair's logical chunks: e from its ring, then the block's own in
// half `half` of wbuf.  A ring of at most nw chunks is rewritten whole by every
// block, from slot 0; a longer one turns: logical chunk j of a block whose first
// chunk is number abs0 of the tile is in slot (abs0 + j) mod e.  lane = chunk.
static_assert(2 * DOG_MAX_RADIUS / 8 + 1 + 12 <= CHUNK_TABLE, "e + warps");
__device__ __forceinline__ void chunk_table(int* table, const PairInfo& U, int nw, int wbuf, int half, int abs0) {
    const int j = threadIdx.x & 31;
    const int slot = U.e > nw ? ring_pos(U, abs0 + j) : j;
    if (j < U.e + nw) table[j] = j < U.e ? U.ring_off + slot * CHUNK : wbuf + (half * nw + j - U.e) * CHUNK;
}

// ---------------------------------------------------------------------------
// Maxima a warp has found, kept in its own shared-memory queue and written out
// (or added to the soft histogram) 32 lanes at a time.
// entry: .x = row (21 bits) | lane << 21 | plane << 26 | strip edge << 31; .y = L_l -
// L_{l+1} there.  Rows count from the tile's first in detection, whose batched
// frames may have any number of rows (their tiles have at most MAX_TILE_ROWS; a base
// that a warp moves along instead cost 11 to 17% of the kernel's time, because the
// compiler then keeps less in registers), and from the frame's first in the soft
// modes, whose frames have at most 65,535.
static_assert(MAX_TILE_ROWS <= 1 << 21, "rows of a queue entry");
__device__ __forceinline__ unsigned q_code(int y, int lane, int l, bool edge) {
    return (unsigned)y | (unsigned)lane << 21 | (unsigned)l << 26 | (unsigned)edge << 31;
}
template <int MODE>
__device__ __forceinline__ int q_base(int y0) { return MODE == MODE_CANDIDATES ? y0 : 0; }

template <int MODE>
__device__ __noinline__ void flush(const FusedParams& p, SmemSmall& ss, int x0, int y_base, int frame,
                                   dog_blob* blobs, int* count, const uint2* queue, int n) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    for (int i0 = 0; i0 < n; i0 += 32) {
        const bool have = i0 + lane < n;
        const uint2 v = have ? queue[i0 + lane] : make_uint2(0u, 0u);
        const int y = y_base + (int)(v.x & ((1 << 21) - 1)), x = x0 + (int)((v.x >> 21) & 31), l = (v.x >> 26) & 31;
        const bool edge = v.x >> 31;
        const float e = __uint_as_float(v.y);
        const float d = __fmul_rn(ss.c[l], e);
        if (MODE == MODE_CANDIDATES) {
            const unsigned mb = __ballot_sync(0xffffffffu, have && !edge), mp = __ballot_sync(0xffffffffu, have && edge);
            int bb = 0, bp = 0;
            if (lane == 0 && mb) bb = atomicAdd(count, __popc(mb));
            if (lane == 0 && mp) bp = atomicAdd(p.pend_count, __popc(mp));
            bb = __shfl_sync(0xffffffffu, bb, 0);
            bp = __shfl_sync(0xffffffffu, bp, 0);
            const int idx = edge ? bp + __popc(mp & lanemask_lt()) : bb + __popc(mb & lanemask_lt());
            if (have && idx >= (edge ? p.pend_cap : p.cap)) {
                atomicCAS(p.status, 0, (int)DOG_ERR_CAPACITY);
            } else if (have && edge) {
                Pending q;
                q.frame = frame; q.x = x; q.y = y; q.level = l; q.response = d;
                p.pend[idx] = q;
            } else if (have) {
                dog_blob bl;
                bl.x = x; bl.y = y; bl.level = l; bl.sigma = ss.sig[l]; bl.response = d;
                blobs[idx] = bl;
            }
        } else if (MODE == MODE_SOFT) {
            int idx = 0;
            if (p.rec != nullptr) {
                const unsigned m = __ballot_sync(0xffffffffu, have);
                if (lane == 0) idx = atomicAdd(p.rec_count + frame, __popc(m));
                idx = __shfl_sync(0xffffffffu, idx, 0) + __popc(m & lanemask_lt());
            }
            const float s = have ? 1.0f / (1.0f + __expf(-(d - p.thr) * p.inv_T)) : 0.0f;
            // one addition per plane and bin: nearly all maxima are of the finest
            // plane, and 32 lanes adding to one word of shared memory take turns
            // (16 frames of 1024 x 1024 with 12 levels: 1657 -> 1549 us)
            for (unsigned left = __ballot_sync(0xffffffffu, have); left;) {
                const int lv = __shfl_sync(0xffffffffu, l, __ffs(left) - 1);
                const bool same = have && l == lv;
                left &= ~__ballot_sync(0xffffffffu, same);
                float t = same ? s : 0.0f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (lane < 2) atomicAdd(&ss.soft[ss.kb[lv][lane]], t * ss.kw[lv][lane]);
            }
            if (have) {
                if (p.rec != nullptr) {
                    if (idx < p.rec_cap) {
                        const float q = s * (1.0f - s) * p.inv_T;
                        dog_soft_max m;
                        m.x = x; m.y = y; m.level = l; m.q = q; m.qe = q * (ss.sg[l] * e); m.s = s;
                        p.rec[(size_t)frame * p.rec_cap + idx] = m;
                    } else {
                        atomicCAS(p.status, 0, (int)DOG_ERR_CAPACITY);
                    }
                }
            }
        }
    }
    __syncwarp();
}

// The 3x3x3 test, plane by plane.  A warp tests the rows one above its own
// (test row t is its row t - 1), so that every neighbour row is its own or one
// of the two the warp above published.
// Everything a warp's test needs to know about its place.
struct TestPlace {
    int y;           // image row of test row 0
    unsigned rows;   // bit t: test row t belongs to the tile
    bool own, edge;  // this lane settles its column; its neighbours lie in the adjacent strip
};

// Candidates of plane l1: cen[t], the plane's centre differences, scaled by c,
// against floor_[t], the largest of the neighbouring maxima and the threshold.
template <int MODE>
__device__ __forceinline__ void settle(const FusedParams& p, SmemSmall& ss, const TileCtx& tc, const TestPlace& at,
                                       int l1, float c, const float (&cen)[8], const float (&floor_)[8], uint2* queue,
                                       int& qn, float (&gp)[8]) {
    bool any = false;
#pragma unroll
    for (int t = 0; t < 8; ++t) any |= __fmul_rn(c, cen[t]) >= floor_[t];
    const bool found = __any_sync(0xffffffffu, any);
    if (MODE != MODE_BWD && !found) return;
    unsigned mask = 0u;
#pragma unroll
    for (int t = 0; t < 8; ++t) mask |= __fmul_rn(c, cen[t]) >= floor_[t] ? 1u << t : 0u;
    mask = at.own ? mask & at.rows : 0u;
    const int lane = threadIdx.x & 31;
    if (MODE == MODE_BWD) {
        // dense dloss/dL rows: A_l = c_l G_l - c_{l-1} G_{l-1}; gp holds c_{l-1} G_{l-1}
        const int x = tc.x0 + lane;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            float g = 0.0f;
            if (mask >> t & 1) {
                const float d = __fmul_rn(c, cen[t]);
                const float s = 1.0f / (1.0f + __expf(-(d - p.thr) * p.inv_T));
                const float G = ss.gk[l1] * s * (1.0f - s) * p.inv_T;
                atomicAdd(&ss.dc[l1], ss.sg[l1] * (G * d / c));
                atomicAdd(&ss.dt[l1], s * ss.gdk[l1]);
                g = ss.sg[l1] * (c * G);
            }
            if (at.own && (at.rows >> t & 1)) {
                const size_t o = ((size_t)l1 * tc.H + at.y + t) * tc.W + x;
                p.A[o] = g - (l1 > 0 ? gp[t] : 0.0f);
                if (l1 == p.P - 1) p.A[o + (size_t)tc.H * tc.W] = -g;
            }
            gp[t] = g;
        }
        return;
    }
    while (__any_sync(0xffffffffu, mask != 0u)) {
        if (qn + 32 > QUEUE_CAP) {
            flush<MODE>(p, ss, tc.x0, q_base<MODE>(tc.y0), tc.frame, tc.blobs, tc.count, queue, qn);
            qn = 0;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, mask != 0u);
        if (mask) {
            const int t = __ffs(mask) - 1;
            mask &= mask - 1;
            float e = cen[0];
#pragma unroll
            for (int u = 1; u < 8; ++u) e = t == u ? cen[u] : e;
            queue[qn + __popc(bal & lanemask_lt())] = make_uint2(q_code(at.y + t - q_base<MODE>(tc.y0), lane, l1, at.edge), __float_as_uint(e));
        }
        qn += __popc(bal);
    }
}

// One plane: its differences of the warp's own rows and of the two rows above
// give the 3x3 maxima of the test rows; then the plane below it in scale, whose
// centre differences are cen, is settled.  Rows and columns outside the frame
// hold -inf.  c > 0 and rounding is monotonic, so the maximum of the scaled
// values is the scaled maximum.  (In the soft modes the caller's sigmas may
// cross, which makes c negative: the differences then carry its sign.)  Lanes 0 and 31 receive their own value from
// the shuffles, which leaves their maximum unchanged: neighbours outside the
// strip are outside the frame or settled elsewhere.  mprev: maxima of plane
// l - 1; mout: of plane l; two[t]: the larger of the last two planes' maxima.
// thr_up: the smallest number above the threshold (D > thr iff D >= thr_up).
template <int MODE>
__device__ __forceinline__ void test_plane(const FusedParams& p, SmemSmall& ss, const TileCtx& tc, const TestPlace& at,
                                           int l, float c, float cprev, const float (&e)[8], float up2, float up1,
                                           const float (&cen)[8], const float (&mprev)[8], float (&mout)[8],
                                           float (&two)[8], float thr_up, uint2* queue, int& qn, float (&gp)[8]) {
    float fl[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const float a = t < 2 ? (t ? up1 : up2) : e[t < 2 ? 0 : t - 2], b = t < 1 ? up1 : e[t < 1 ? 0 : t - 1];
        const float v = fmaxf(e[t], fmaxf(a, b));
        const float vl = __shfl_up_sync(0xffffffffu, v, 1), vr = __shfl_down_sync(0xffffffffu, v, 1);
        mout[t] = __fmul_rn(c, fmaxf(v, fmaxf(vl, vr)));
        fl[t] = fmaxf(thr_up, fmaxf(mout[t], two[t]));
        two[t] = fmaxf(mprev[t], mout[t]);
    }
    if (l > 0) settle<MODE>(p, ss, tc, at, l - 1, cprev, cen, fl, queue, qn, gp);
}

// ---------------------------------------------------------------------------
// Input rows y .. y + 7 into the buffer's slots `slot` .. (modulo CIN), by one
// warp: lane x takes columns x, x + 32, ...; four rows by three columns of loads
// in flight before any is converted and stored (more would cost the passes
// around it their registers).
__device__ __forceinline__ void load8(SmemSmall& ss, int R, int y, float* in, int slot, int CIN, int S) {
    const PixelSource px = ss.px;
    const int lane = threadIdx.x & 31, ncols = TX + 2 * R;
    bool bad = false;
#pragma unroll 1
    for (int c0 = lane; c0 < ncols; c0 += 96) {
        int xr[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) xr[k] = refl(px.x0 - R + min(c0 + 32 * k, ncols - 1), px.W);
        int s = slot;
#pragma unroll 1
        for (int j0 = 0; j0 < 8; j0 += 4) {
            unsigned v[4][3];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int yr = refl(y + j0 + j, px.H);
#pragma unroll
                for (int k = 0; k < 3; ++k) v[j][k] = load_raw(px.img, px.dtype, px.pitch, yr, xr[k]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float* dst = in + s * S + c0;
                s = s + 1 == CIN ? 0 : s + 1;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float v1 = raw_to_px(v[j][k], px.dtype, px.st_lo, px.st_hi, px.st_rcp);
                    if (c0 + 32 * k < ncols) dst[32 * k] = v1;
                    bad |= !(fabsf(v1) < HUGE_PX);
                }
            }
        }
    }
    if (bad) ss.careful = 1;
}

template <int NW, int MODE, bool BATCHED>
__device__ __forceinline__ void process_tile(const FusedParams& p, float* sm, SmemSmall& ss, const TileCtx& tc) {
    constexpr bool CT = MODE == MODE_CANDIDATES || MODE == MODE_DUMP;   // taps in the kernel's parameters
    constexpr bool TEST = MODE != MODE_DUMP;
    constexpr int MBK = 8 * NW;   // rows of a block
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rho = lane >> 2;
    const int R = p.R, S = p.in_stride, CIN = p.in_rows, n = p.n_pairs, off = p.lev_off;
    float* in = sm + p.in_off;
    float* wbuf = sm + p.w_off;
    float* xch = sm + p.x_off;      // [parity][plane of the pair][warp][2 rows][32]
    float* eh = sm + p.e_off;       // [plane][2 rows][32]: the last two rows of the block before
    uint2* queue = reinterpret_cast<uint2*>(sm + p.q_off) + warp * QUEUE_CAP;
    int* tables = reinterpret_cast<int*>(sm + p.c_off);   // [half of wbuf][pair][CHUNK_TABLE]
    const Taps<CT> tap{p, reinterpret_cast<const float4*>(sm + p.t_off)};
    int qn = 0;

    // rows computed: yb0 .. ylast (one above and one below the band, inside the
    // frame); the test of a block's last row waits for the next block
    const int yb0 = TEST && tc.y0 > 0 ? tc.y0 - 1 : tc.y0;
    const int ylast = TEST ? min(tc.y1, tc.H - 1) : tc.y1 - 1;
    const int nblk = ((TEST ? tc.y1 + 1 : tc.y1) - yb0 + MBK - 1) / MBK;
    const int gx = tc.x0 + lane;
    const bool col_ok = gx >= 0 && gx < tc.W;
    const bool overlap = !BATCHED && p.overlap;   // (single-frame launches only)
    TestPlace at;
    at.own = col_ok && (!overlap || (lane >= 1 && lane <= TX - 2));
    at.edge = !overlap && ((lane == 0 && tc.x0 > 0) || (lane == TX - 1 && gx + 1 < tc.W));
    const bool cut = tc.x0 < 0 || tc.x0 + TX > tc.W;   // columns outside the frame
    // soft modes keep every maximum
    const float thr_up = MODE == MODE_CANDIDATES ? p.thr_up : -FLT_MAX;

    int base = 0;            // input slot of image row yb + dmin, yb the current block's
    // this lane's input row of the warp's chunk for pair U
    auto row_of = [&](const PairInfo& U) {
        int s = base + U.delta - p.dmin + 8 * warp + rho;
        s -= s >= CIN ? CIN : 0;
        return in + s * S;
    };
    // warm-up: the horizontal sums of the e chunks above the first block, in
    // blocks of their own (warp w's chunk is chunk e - NW m + w of the ring)
    int emax = 0;
    for (int q = 0; q < n; ++q) emax = max(emax, (int)p.pairs[q].e);
    const int nwarm = (emax + NW - 1) / NW;
    if (tid == 0) {
        ss.careful = 0;
        // (field by field: nvcc 13.0 turns a copy of a whole struct into a copy of the
        // kernel parameters its first fields came from)
        ss.px.img = tc.img;
        ss.px.dtype = tc.dtype;
        ss.px.H = tc.H;
        ss.px.W = tc.W;
        ss.px.pitch = tc.pitch;
        ss.px.st_lo = tc.st_lo;
        ss.px.st_hi = tc.st_hi;
        ss.px.st_rcp = tc.st_rcp;
        ss.px.x0 = tc.x0;
    }
    __syncthreads();
    for (int r = 8 * warp; r < CIN; r += MBK) {   // (the last group's rows past CIN go to the first slots again)
        const int at0 = min(r, CIN - 8);
        load8(ss, R, yb0 - MBK * nwarm + p.dmin + at0, in, at0, CIN, S);
    }
    for (int q = warp; q < 2 * n; q += NW)
        chunk_table(tables + q * CHUNK_TABLE, p.pairs[q < n ? q : q - n], NW, p.w_off, q >= n, 0);
    __syncthreads();
    for (int m = nwarm; m > 0; --m) {
        for (int q = 0; q < n; ++q) {
            const PairInfo& U = p.pairs[q];
            const int c = U.e - NW * m + warp;
            if (c >= 0 && c < U.e)
                hpass(U, sm, row_of(U), R, sm + U.ring_off + c * CHUNK, tap, ss.careful != 0);
        }
        __syncthreads();
        int s = base + 8 * warp;   // over the rows no longer read
        load8(ss, R, yb0 - MBK * (m - 1) + p.dmax + 8 * warp, in, s - (s >= CIN ? CIN : 0), CIN, S);
        base = (base + MBK) % CIN;
        __syncthreads();
    }
    hpass(p.pairs[0], sm, row_of(p.pairs[0]), R, wbuf + warp * CHUNK, tap, ss.careful != 0);
    __syncthreads();

    // test state between planes: the scaled 3x3 maxima m1 of the last plane (m2 is
    // its partner, so that no maxima are copied), the larger of the last two
    // planes' maxima, and the last plane's centre differences e1, which are
    // settled as soon as the next plane's maxima exist; gp: the backward mode's
    // c G of the plane before
    float Lp[8], eA[8], eB[8], e1[8], m1[8], m2[8], two[8], gp[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        m1[k] = m2[k] = two[k] = e1[k] = eA[k] = eB[k] = -INFINITY;
        Lp[k] = gp[k] = 0.0f;
    }
    int par = 0;     // buffer half of the current interval's pair
    int abs0 = 0;    // chunks before the current block (ring slots are taken modulo e)
    at.rows = 0u;
    for (int b = 0;; ++b) {   // block nblk: only the last planes' test
        const int yb = yb0 + MBK * b;
        const bool last = b + 1 == nblk;
        const int yw = yb + 8 * warp;             // this warp's first row
        const bool act = yw <= ylast;             // it has rows to compute
        const bool inside = yw + 7 < tc.H && !cut;
        for (int q = 0; q < n; ++q) {
            const PairInfo& U = p.pairs[q];
            const bool careful = ss.careful != 0;
            const bool some = q > 0 || b > 0;      // there was an interval before
            const int lq = q ? q - 1 : n - 1;      // and this was its pair
            if (TEST && q == 1) {   // the planes tested from here on are this block's
                at.y = yw - 1;
                const int lo = max(tc.y0 - at.y, 0), hi = min(tc.y1 - at.y, 8);   // test rows lo .. hi-1
                at.rows = hi > lo && (MODE != MODE_CANDIDATES || p.thr < INFINITY) ? ((1u << hi) - 1u) & ~((1u << lo) - 1u) : 0u;
            }
            // 1. keep the chunk of the pair before for its next block (the last e
            // chunks, in the slots after the block's); stored after the test
            const PairInfo& V = p.pairs[lq];
            const int kc = warp - (NW - V.e);
            const bool keep = some && kc >= 0;
            float4 kept[CHUNK / 128];
            if (keep) {
                const float4* s4 = reinterpret_cast<const float4*>(wbuf + (par ^ 1) * (NW * CHUNK) + warp * CHUNK);
#pragma unroll
                for (int i = 0; i < CHUNK / 128; ++i) kept[i] = s4[i * 32 + lane];
                const int slot = V.e > NW ? ring_pos(V, (q ? abs0 + NW : abs0) + kc) : kc;
                float4* d4 = reinterpret_cast<float4*>(sm + V.ring_off + slot * CHUNK);
#pragma unroll
                for (int i = 0; i < CHUNK / 128; ++i) d4[i * 32 + lane] = kept[i];
            }
            __syncwarp();
            // 2. horizontal pass of the next pair (the last pair's interval does the
            // next block's first one below): half of the warps of each scheduler run
            // it before the test, so that the test's comparisons meet other warps' FMAs
            auto ahead = [&]() {
                const PairInfo& N = p.pairs[q + 1];
                hpass(N, sm, row_of(N), R, wbuf + (par ^ 1) * (NW * CHUNK) + warp * CHUNK, tap, careful);
            };
            const bool go = q + 1 < n && act && b < nblk;
            if (go && (warp & 4)) ahead();
            // 3. the planes published in the interval before
            if (TEST && some) {
                const bool first = q ? b == 0 : b == 1;   // they are of the tile's first block
                const float* xr = xch + (par ^ 1) * (2 * NW * 64);
                float upA1 = -INFINITY;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int l = 2 * lq - 1 - off + s;
                    if (l < 0) continue;
                    const float* src = warp ? xr + (s * NW + warp - 1) * 64 : eh + l * 64;
                    float up2 = src[lane], up1 = src[32 + lane];
                    if (warp == 0) {
                        if (first) up2 = up1 = -INFINITY;
                        const float* lw = xr + (s * NW + NW - 1) * 64;
                        eh[l * 64 + lane] = lw[lane];
                        eh[l * 64 + 32 + lane] = lw[32 + lane];
                    }
                    const float c = CT ? p.cn[l] : ss.c[l], cp = CT ? p.cn[max(l - 1, 0)] : ss.c[max(l - 1, 0)];
                    if (s == 0) {
                        upA1 = up1;
                        test_plane<MODE>(p, ss, tc, at, l, c, cp, eA, up2, up1, e1, m1, m2, two, thr_up, queue, qn, gp);
                    } else {
                        const float cen[8] = {upA1, eA[0], eA[1], eA[2], eA[3], eA[4], eA[5], eA[6]};
                        test_plane<MODE>(p, ss, tc, at, l, c, cp, eB, up2, up1, cen, m2, m1, two, thr_up, queue, qn, gp);
                        e1[0] = up1;
#pragma unroll
                        for (int t = 1; t < 8; ++t) e1[t] = eB[t - 1];
                    }
                }
                if (q == 0) {   // the last plane has nothing above it
#pragma unroll
                    for (int t = 0; t < 8; ++t) two[t] = fmaxf(thr_up, two[t]);
                    settle<MODE>(p, ss, tc, at, p.P - 1, CT ? p.cn[p.P - 1] : ss.c[p.P - 1], e1, two, queue, qn, gp);
#pragma unroll
                    for (int t = 0; t < 8; ++t) m1[t] = m2[t] = two[t] = -INFINITY;
                }
            }
            if (b == nblk) {
                if (TEST && qn) flush<MODE>(p, ss, tc.x0, q_base<MODE>(tc.y0), tc.frame, tc.blobs, tc.count, queue, qn);
                __syncthreads();
                return;
            }
            if (go && !(warp & 4)) ahead();
            // a turning ring: the pair's chunk table for the next block
            if (V.e > NW && some && warp == 0) chunk_table(tables + (((par ^ 1 ^ n) & 1) * n + lq) * CHUNK_TABLE, V, NW, p.w_off, (par ^ 1 ^ n) & 1, q ? abs0 + NW : abs0);
            // 4. vertical pass and the differences it completes
            if (act) {
                float2 acc[8];
                vpass(U, sm, tables + (par * n + q) * CHUNK_TABLE + warp, tap, careful, acc);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    eA[k] = __fsub_rn(Lp[k], acc[k].x);
                    eB[k] = __fsub_rn(acc[k].x, acc[k].y);
                    Lp[k] = acc[k].y;
                }
                if ((MODE == MODE_SOFT || MODE == MODE_BWD) && ss.flip) {
                    const int l = 2 * q - 1 - off;
                    const float sa = ss.sg[max(l, 0)], sb = ss.sg[max(l + 1, 0)];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        eA[k] *= sa;
                        eB[k] *= sb;
                    }
                }
                if (MODE == MODE_DUMP) {
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        const int l = 2 * q - 1 - off + s;
                        if (l < 0 || !at.own) continue;
                        const float c = p.cn[l];
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (yw + k < tc.y1)
                                p.dump[((size_t)l * tc.H + yw + k) * tc.W + gx] = __fmul_rn(c, s ? eB[k] : eA[k]);
                    }
                } else if (!inside) {   // rows and columns outside the frame do not count
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (yw + k >= tc.H || !col_ok) eA[k] = eB[k] = -INFINITY;
                }
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k) eA[k] = eB[k] = -INFINITY;
            }
            if (TEST) {
                float* xw = xch + par * (2 * NW * 64) + warp * 64 + lane;
                xw[0] = eA[6];
                xw[32] = eA[7];
                xw[NW * 64] = eB[6];
                xw[NW * 64 + 32] = eB[7];
            }
            if (q + 1 == n && !last) {
                // the next block's input rows, over the rows no longer read
                int s = base + 8 * warp;
                s -= s >= CIN ? CIN : 0;
                load8(ss, R, yb + MBK + p.dmax + 8 * warp, in, s, CIN, S);
                __syncthreads();
                base = (base + MBK) % CIN;
                if (yw + MBK <= ylast)
                    hpass(p.pairs[0], sm, row_of(p.pairs[0]), R,
                          wbuf + (par ^ 1) * (NW * CHUNK) + warp * CHUNK, tap, ss.careful != 0);
            }
            __syncthreads();
            par ^= 1;
        }
        abs0 += NW;
    }
}

template <int NW, int MODE, bool BATCHED>
__global__ void __launch_bounds__(NW * 32, 1) dog_fused_kernel(const __grid_constant__ FusedParams p) {
    constexpr int NTHREADS = NW * 32;
    constexpr bool SOFT = MODE == MODE_SOFT || MODE == MODE_BWD;
    extern __shared__ float4 dyn4[];
    float* sm = reinterpret_cast<float*>(dyn4);
    __shared__ SmemSmall ss;
    const int tid = threadIdx.x;
    // zero-weight padding taps may read input-row columns past the loaded ones,
    // and those must be finite
    {
        const int c0 = TX + 2 * p.R, nc = p.in_stride - c0;
        for (int q = tid; q < p.in_rows * nc; q += NTHREADS) sm[p.in_off + q / nc * p.in_stride + c0 + q % nc] = 0.0f;
    }
    for (int q = tid; q < p.P; q += NTHREADS) {
        ss.c[q] = SOFT ? fabsf(p.c[q]) : p.c[q];
        ss.sig[q] = p.c[p.P + q];
        if (SOFT) ss.sg[q] = copysignf(1.0f, p.c[q]);
    }
    if (SOFT) {
        bool neg = false;
        for (int q = tid; q < p.P; q += NTHREADS) neg |= p.c[q] < 0.0f;
        ss.flip = __syncthreads_or(neg);
        float4* t4 = reinterpret_cast<float4*>(sm + p.t_off);
        const float4* w4 = reinterpret_cast<const float4*>(p.w);
        for (int q = tid; q < p.n_taps4; q += NTHREADS) t4[q] = w4[q];
        for (int q = tid; q < p.nbins; q += NTHREADS) ss.soft[q] = 0.0f;
        for (int l = tid; l < p.P; l += NTHREADS) {
            float gk = 0.0f, gdk = 0.0f;
            int nb = 0;
            ss.kb[l][0] = 0; ss.kb[l][1] = 0; ss.kw[l][0] = 0.0f; ss.kw[l][1] = 0.0f;
            for (int b = 0; b < p.nbins; ++b) {
                const float k = p.kappa[l * p.nbins + b];
                if (p.gH) {
                    gk += p.gH[b] * k;
                    gdk += p.gH[b] * p.dkappa[l * p.nbins + b];
                }
                if (k != 0.0f && nb < 2) { ss.kb[l][nb] = b; ss.kw[l][nb] = k; ++nb; }
            }
            ss.gk[l] = gk; ss.gdk[l] = gdk; ss.dc[l] = 0.0f; ss.dt[l] = 0.0f;
        }
    }

    if (!BATCHED) {
        // single frame: blockIdx.x enumerates (strip, band)
        __syncthreads();
        TileCtx tc;
        int tile = blockIdx.x, frame = 0;
        if (MODE == MODE_SOFT) {   // of a batch of equal frames, frame after frame
            frame = tile / (p.n_strips * p.n_bands);
            tile -= frame * (p.n_strips * p.n_bands);
        }
        tc.img = MODE == MODE_SOFT ? static_cast<const float*>(p.img) + frame * p.frame_stride : p.img;
        tc.dtype = p.dtype; tc.H = p.H; tc.W = p.W; tc.pitch = p.pitch; tc.frame = frame;
        tc.st_lo = tc.dtype == DTYPE_U16_STRETCH ? p.lohi[0] : 0;
        tc.st_hi = tc.dtype == DTYPE_U16_STRETCH ? p.lohi[1] : 0;
        tc.st_rcp = stretch_rcp(tc.st_lo, tc.st_hi);
        const int band = tile / p.n_strips, strip = tile - band * p.n_strips;
        tc.x0 = strip * p.strip_step + p.strip_x0;
        tc.y0 = band * p.band;
        tc.y1 = min(p.H, tc.y0 + p.band);
        tc.blobs = p.blobs;
        tc.count = p.count;
        process_tile<NW, MODE, BATCHED>(p, sm, ss, tc);
    } else {
        const long long n_tiles = p.ntiles_dev ? *p.ntiles_dev : p.n_tiles;
        for (;;) {
            __syncthreads();
            if (tid == 0) ss.tile = atomicAdd(p.tile_counter, 1);
            __syncthreads();
            const long long t = ss.tile;
            if (t >= n_tiles) break;
            int lo = 0, hi = p.n_frames - 1;
            while (lo < hi) {   // last frame whose tile_begin <= t
                const int mid = (lo + hi + 1) >> 1;
                if (p.frames[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
            }
            const FrameDesc f = p.frames[lo];
            const int local = (int)(t - f.tile_begin);
            TileCtx tc;
            tc.img = f.img; tc.dtype = f.dtype; tc.H = f.h; tc.W = f.w; tc.pitch = f.pitch; tc.frame = lo;
            tc.st_lo = tc.dtype == DTYPE_U16_STRETCH ? p.lohi[2 * lo] : 0;
            tc.st_hi = tc.dtype == DTYPE_U16_STRETCH ? p.lohi[2 * lo + 1] : 0;
            tc.st_rcp = stretch_rcp(tc.st_lo, tc.st_hi);
            tc.x0 = (local % f.n_strips) * TX;
            const int band = local / f.n_strips;
            const int bh = f.band;
            tc.y0 = band * bh;
            tc.y1 = min(f.h, tc.y0 + bh);
            tc.blobs = p.blobs + f.blob_off;
            tc.count = p.count + lo;
            process_tile<NW, MODE, BATCHED>(p, sm, ss, tc);
        }
        if (tid == 0) {
            __threadfence();
            const int d = atomicAdd(p.done_counter, 1);
            if (d == (int)gridDim.x - 1) {
                atomicExch(p.tile_counter, 0);
                atomicExch(p.done_counter, 0);
            }
        }
    }

    if (SOFT) {
        __syncthreads();
        if (MODE == MODE_SOFT) {
            for (int q = tid; q < p.nbins; q += NTHREADS)
                if (ss.soft[q] != 0.0f) atomicAdd(&p.soft_out[q], ss.soft[q]);
        } else {
            for (int q = tid; q < p.P; q += NTHREADS) {
                if (ss.dc[q] != 0.0f) atomicAdd(&p.dc_acc[q], (double)ss.dc[q]);
                if (ss.dt[q] != 0.0f) atomicAdd(&p.dt_acc[q], (double)ss.dt[q]);
            }
        }
    }
}

// The dynamic shared-memory limit is raised once per device and kernel form
// (not on every launch, so launches can be captured into CUDA graphs), to the
// most that any handle asks for: handles of other ladders on other host threads
// launch the same forms, and setting one size twice is harmless.
template <int NW, int MODE, bool BATCHED>
static cudaError_t launch_form(const FusedParams& p, int grid, cudaStream_t s) {
    static std::atomic<bool> raised[64];
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!raised[dev & 63].load(std::memory_order_acquire)) {
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(dog_fused_kernel<NW, MODE, BATCHED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     optin - SMEM_RESERVE);
        if (e != cudaSuccess) return e;
        raised[dev & 63].store(true, std::memory_order_release);
    }
    dog_fused_kernel<NW, MODE, BATCHED><<<grid, NW * 32, p.smem_bytes, s>>>(p);
    return cudaGetLastError();
}

// All forms of one warp count (each translation unit instantiates one).
cudaError_t launch_fused_w12(const FusedParams& p, int grid, cudaStream_t s);
cudaError_t launch_fused_w10(const FusedParams& p, int grid, cudaStream_t s);
cudaError_t launch_fused_w8(const FusedParams& p, int grid, cudaStream_t s);
cudaError_t launch_fused_w4(const FusedParams& p, int grid, cudaStream_t s);
cudaError_t launch_fused_w3(const FusedParams& p, int grid, cudaStream_t s);
cudaError_t launch_fused_w2(const FusedParams& p, int grid, cudaStream_t s);
#define DOG_FUSED_FORMS(NW)                                                                       \
    cudaError_t launch_fused_w##NW(const FusedParams& p, int grid, cudaStream_t s) {              \
        if (p.frames != nullptr) return launch_form<NW, MODE_CANDIDATES, true>(p, grid, s);       \
        switch (p.mode) {                                                                         \
            case MODE_CANDIDATES: return launch_form<NW, MODE_CANDIDATES, false>(p, grid, s);     \
            case MODE_DUMP: return launch_form<NW, MODE_DUMP, false>(p, grid, s);                 \
            case MODE_SOFT: return launch_form<NW, MODE_SOFT, false>(p, grid, s);                 \
            default: return launch_form<NW, MODE_BWD, false>(p, grid, s);                         \
        }                                                                                         \
    }

}  // namespace dogk

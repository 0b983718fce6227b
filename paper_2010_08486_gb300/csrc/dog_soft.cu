// Differentiable soft blob-volume histogram and its backward pass (sm_103a).
//
// Not in the paper: a smooth relaxation of the volume histogram of Sec. 4 so
// that the sigma ladder can be tuned by gradient descent towards a steering
// objective.  Over the hard 3x3x3 local maxima v of D (no threshold),
//   H_b = sum_v s_v kappa_b(t_l),   s_v = sigmoid((D_v - thr) / T),
// t_l the normalised log volume of plane l against the handle's ladder ends
// and kappa_b a triangular weight one bin wide.  With the mask and radii
// held fixed, for dloss/dH = gH:
//   G_v = (sum_b gH_b kappa_b(t_l)) s_v (1 - s_v) / T          (dloss/dD_v)
//   A_i = c_i G_i - c_{i-1} G_{i-1}                             (dloss/dL_i)
//   dloss/dI = sum_i B_i^T A_i,     B_i = row blur o column blur (reflect)
//   dloss/dsigma_i = <B_y^T A_i, B_x' I> + <B_y'^T A_i, B_x I>  (kernel shape)
//                  + dloss/dc terms + dloss/dt terms.
// Every B_i is symmetric: its kernel is even and the boundary reflects about
// the half sample, so B_i^T A is the blur of A itself with the same boundary.
// Two backward paths.  From a record of the forward's maxima (soft forward
// with `rec`): A is zero outside the maxima's voxels, so dloss/dI is gathered
// tile by tile from the maxima whose windows reach it, and the kernel-shape
// term is evaluated at the maxima as sum_v A_i(v) dL_i/dsigma_i(v); no plane of
// A and no blur level is formed.  Without a record: the fused kernel (MODE_BWD)
// recomputes the L_i and writes A densely, two passes blur it, and the
// kernel-shape term is the two inner products above.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "dog_internal.cuh"

namespace dogk {

const FusedParams& handle_base(const dog_handle* h);
int handle_K(const dog_handle* h);
int handle_P(const dog_handle* h);
const std::vector<int>& handle_radii(const dog_handle* h);
const std::vector<double>& handle_sigmas(const dog_handle* h);
const dog_config& handle_cfg(const dog_handle* h);
int handle_band(const dog_handle* h);
int handle_w_total(const dog_handle* h);
int handle_sms(const dog_handle* h);
int handle_wait_limit(const dog_handle* h);
int pick_band(const FusedParams& b, int num_sms, int H, int n_strips, int asked);
const std::vector<LevelInfo>& handle_levels(const dog_handle* h);
void handle_tap_slot(const dog_handle* h, int i, int* base, int* lead);
int* handle_status(dog_handle* h);
void*& handle_soft_ws(dog_handle* h);
cudaError_t timed_fused(dog_handle* h, const FusedParams& p, int grid, cudaStream_t s);

struct SoftWS {
    int H = 0, W = 0;
    float* w = nullptr;       // taps from the device sigmas, plain table
    float* dw = nullptr;      // their derivative wrt sigma
    float* wp = nullptr;      // the taps in the fused kernel's pair layout
    float* c = nullptr;       // P coefficients then P sigmas
    float* kappa = nullptr;   // P x nbins
    float* dkappa = nullptr;  // P x nbins
    float* gk = nullptr;      // P sums gH . kappa_l, then P sums gH . dkappa_l
    float* wpad = nullptr;    // the taps with TAP_PAD zeros around each level's
    float4* wt = nullptr;     // per plane and window offset: taps and their derivatives of both its levels
    float* A = nullptr;       // K x H x W
    void* lists = nullptr;    // the record path's lists (see Lists) of n_lists frames
    int n_lists = 0;
    void* old_lists[8] = {};  // outgrown (see list_frames)
    int n_old = 0;
    int* flags = nullptr;     // per listed frame: FrameFlags; then the grid barrier's counter
    int dense_grid = 0;       // co-resident CTAs of the dense record kernel (0: not asked yet)
    float* Y = nullptr;       // K x H x W
    float* Yd = nullptr;      // K x H x W
    double* acc = nullptr;    // dc (P), dt (P), dw (K), ACC_COPIES times
    float* last_sig = nullptr;   // the sigmas the tables were last built from (NaN: none)
};

void soft_free(dog_handle* h) {
    SoftWS* ws = static_cast<SoftWS*>(handle_soft_ws(h));
    if (!ws) return;
    void* ptrs[] = {ws->w, ws->dw, ws->wp, ws->c, ws->kappa, ws->dkappa, ws->gk, ws->wpad, ws->wt, ws->A, ws->lists, ws->flags, ws->Y, ws->Yd, ws->acc, ws->last_sig};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    for (int i = 0; i < ws->n_old; ++i) cudaFree(ws->old_lists[i]);
    delete ws;
    handle_soft_ws(h) = nullptr;
}

// CTAs of the record pass spread their atomics over copies of the sums.
constexpr int ACC_COPIES = 16;

// The record path lists the maxima by cells of CELL x CELL pixels.  A cell has
// CELL_SLOTS places for the maxima of narrow planes (nearly all; two to a cell in
// a dense frame), which a reader fetches side by side; those of wider planes,
// and what does not fit, are linked.  A frame that overflows the entries or links
// more than CHAIN_MAX to a cell takes the dense form.
constexpr int CELL_SHIFT = 3, CELL_SLOTS = 8, CHAIN_MAX = 64, NARROW_R = 7;
__host__ __device__ static inline int cells(int n) { return (n + (1 << CELL_SHIFT) - 1) >> CELL_SHIFT; }

struct Lists {
    int4* slots;      // cells x CELL_SLOTS: x, y * 32 + plane, A_l there
    int4* ent;        // ent_cap: the same, and the next entry
    int* count;       // cells: maxima of narrow planes
    int* linked;      // cells: entries linked
    int* head;        // cells: first of them, -1 for none
    int n_cells, ent_cap;
    long long ints;   // ints of a frame
};
// Words of a listed frame.  The record and the tile kernel each ask for the dense
// form in a word of its own, so that the tile kernel reads none that its own CTAs
// write (the warps of one would not see the same value).
struct FrameFlags {
    int dense;    // set by the record kernel: the lists do not hold the frame
    int linked;   // entries linked
    int tiles;    // set by the tile kernel: a tile is reached by too many pairs
};
constexpr int LIST_FRAMES = 64;                      // frames of a batch listed at a time, at most,
static_assert(LIST_FRAMES <= 64, "seven growths: SoftWS::old_lists");
constexpr size_t LIST_BYTES = (size_t)256 << 20;     // and the lists' size (one frame's always fit)

// Frame f's lists (all of a frame's arrays lie together).
__host__ __device__ static inline Lists frame_lists(void* base, int H, int W, int f) {
    Lists a;
    a.n_cells = cells(H) * cells(W);
    a.ent_cap = (int)((long long)H * W / 16) + 4096;
    a.ints = 4LL * a.n_cells * CELL_SLOTS + 4LL * a.ent_cap + ((3LL * a.n_cells + 3) & ~3LL);
    int* b = static_cast<int*>(base) + f * a.ints;
    a.slots = reinterpret_cast<int4*>(b);
    a.ent = a.slots + (long long)a.n_cells * CELL_SLOTS;
    a.count = reinterpret_cast<int*>(a.ent + a.ent_cap);
    a.linked = a.count + a.n_cells;
    a.head = a.linked + a.n_cells;
    return a;
}

// Plane l's window holds the kernels of both its levels; offset of its taps.
static int plane_radius(const dog_handle* h, int l) {
    return std::max(handle_levels(h)[l].r, handle_levels(h)[l + 1].r);
}

// Place of level i's taps among the padded ones (i = K: their number).
constexpr int TAP_PAD = 32;
static int pad_offset(const dog_handle* h, int i) {
    int n = TAP_PAD;   // neighbours share the zeros between them
    for (int k = 0; k < i; ++k) n += 2 * handle_levels(h)[k].r + 1 + TAP_PAD;
    return n;
}

static int soft_ws(dog_handle* h, int H, int W, SoftWS** out) {
    SoftWS* ws = static_cast<SoftWS*>(handle_soft_ws(h));
    if (ws && ws->H >= H && ws->W >= W) { *out = ws; return DOG_OK; }
    if (ws) { cudaDeviceSynchronize(); soft_free(h); }
    ws = new SoftWS();
    handle_soft_ws(h) = ws;
    const FusedParams& b = handle_base(h);
    const int K = b.K, P = b.P, nb = handle_cfg(h).nbins;
    const size_t plane = (size_t)H * W;
    cudaError_t e = cudaSuccess;
    auto ok = [&](cudaError_t x) { if (e == cudaSuccess) e = x; };
    ok(cudaMalloc(&ws->w, sizeof(float) * handle_w_total(h)));
    ok(cudaMalloc(&ws->dw, sizeof(float) * handle_w_total(h)));
    ok(cudaMalloc(&ws->wp, sizeof(float4) * b.n_taps4));
    if (e == cudaSuccess) ok(cudaMemset(ws->wp, 0, sizeof(float4) * b.n_taps4));   // padding taps stay zero
    ok(cudaMalloc(&ws->c, sizeof(float) * 2 * P));
    ok(cudaMalloc(&ws->kappa, sizeof(float) * P * nb));
    ok(cudaMalloc(&ws->dkappa, sizeof(float) * P * nb));
    int n_wt = 0;
    for (int l = 0; l < P; ++l) n_wt += 2 * plane_radius(h, l) + 1;
    ok(cudaMalloc(&ws->wt, sizeof(float4) * n_wt));
    ok(cudaMalloc(&ws->gk, sizeof(float) * 2 * P));
    ok(cudaMalloc(&ws->wpad, sizeof(float) * pad_offset(h, K)));
    if (e == cudaSuccess) ok(cudaMemset(ws->wpad, 0, sizeof(float) * pad_offset(h, K)));
    ok(cudaMalloc(&ws->A, sizeof(float) * plane * K));
    ok(cudaMalloc(&ws->lists, sizeof(int) * frame_lists(nullptr, H, W, 0).ints));
    ws->n_lists = 1;
    ok(cudaMalloc(&ws->flags, sizeof(FrameFlags) * LIST_FRAMES + sizeof(int)));
    ok(cudaMalloc(&ws->Y, sizeof(float) * plane * K));
    ok(cudaMalloc(&ws->Yd, sizeof(float) * plane * K));
    ok(cudaMalloc(&ws->acc, sizeof(double) * ACC_COPIES * (2 * P + K)));
    ok(cudaMalloc(&ws->last_sig, sizeof(float) * K));
    if (e == cudaSuccess) ok(cudaMemset(ws->last_sig, 0xff, sizeof(float) * K));   // NaN: tables not built
    if (e != cudaSuccess) {
        soft_free(h);
        return e == cudaErrorMemoryAllocation ? DOG_ERR_NOMEM : DOG_ERR_CUDA;
    }
    ws->H = H;
    ws->W = W;
    *out = ws;
    return DOG_OK;
}

// ---------------------------------------------------------------------------
struct SoftPrep {
    const float* sig;
    int K, P, nbins, norm;
    int r[MAX_LEVELS];
    int woff[MAX_LEVELS];
    int tpad[MAX_LEVELS];
    int pbase[MAX_LEVELS], plead[MAX_LEVELS];   // place of the level's taps in the pair table
    int wtoff[MAX_LEVELS];                      // place of plane l's taps in wt
    double lref0, lrefP;   // ln sigma of the reference ladder's first / last DoG plane
    float* w;
    float* dw;
    float* wp;
    float* c;
    float* kappa;
    float* dkappa;
    float* last_sig;
    float4* wt;
    float* wpad;
    int padoff[MAX_LEVELS];
    const float* gH;   // backward: dloss/dH (nullptr in the forward)
    float* gk;
    int* zero;         // counters to clear
    int n_zero;
    double* acc;       // sums to clear
    int n_acc;
    void* lists;       // lists of n_lists frames of H x W to empty
    int n_lists, H, W;
};

constexpr int PREP_THREADS = 512, PREP_CELLS = 8 * PREP_THREADS;

__device__ void soft_tables(const SoftPrep& p) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < p.K; i += PREP_THREADS / 32) {
        const double s = (double)p.sig[i];
        const int r = p.r[i];
        double z = 0.0, m2 = 0.0;
        for (int j = -r + lane; j <= r; j += 32) {
            const double e = exp(-(double)j * j / (2.0 * s * s));
            z += e;
            m2 += e * (double)j * j;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            z += __shfl_xor_sync(0xffffffffu, z, o);
            m2 += __shfl_xor_sync(0xffffffffu, m2, o);
        }
        m2 /= z;
        // full taps t = 0..2r (offset t - r), zero-padded to tpad
        for (int t = lane; t < p.tpad[i]; t += 32) {
            const int j = t - r;
            float wv = 0.0f, dv = 0.0f;
            if (t <= 2 * r) {
                const double wj = exp(-(double)j * j / (2.0 * s * s)) / z;
                wv = (float)wj;
                dv = (float)(wj * ((double)j * j - m2) / (s * s * s));
            }
            p.w[p.woff[i] + t] = wv;
            p.dw[p.woff[i] + t] = dv;
            if (t <= 2 * r) {
                p.wp[p.pbase[i] + 2 * (t + p.plead[i])] = wv;
                p.wpad[p.padoff[i] + t] = wv;
            }
        }
    }
    for (int l = threadIdx.x; l < p.P; l += blockDim.x) {
        const double s0 = (double)p.sig[l], s1 = (double)p.sig[l + 1];
        p.c[l] = (float)(p.norm == DOG_NORM_PAPER ? s0 : s0 / (s1 - s0));
        p.c[p.P + l] = (float)s0;
        const double t = (log(s0) - p.lref0) / (p.lrefP - p.lref0);
        const double lo = 0.5 / p.nbins, hi = 1.0 - 0.5 / p.nbins;
        const bool clamped = (t < lo) || (t > hi);
        const double tc = fmin(fmax(t, lo), hi);
        for (int b = 0; b < p.nbins; ++b) {
            const double u = (double)p.nbins * tc - ((double)b + 0.5);
            const double a = fabs(u);
            p.kappa[l * p.nbins + b] = a < 1.0 ? (float)(1.0 - a) : 0.0f;
            const double sg = u > 0.0 ? 1.0 : (u < 0.0 ? -1.0 : 0.0);
            p.dkappa[l * p.nbins + b] = (a < 1.0 && !clamped) ? (float)(-(double)p.nbins * sg) : 0.0f;
        }
    }
    for (int i = threadIdx.x; i < p.K; i += blockDim.x) p.last_sig[i] = p.sig[i];
    __syncthreads();
    for (int l = warp; l < p.P; l += PREP_THREADS / 32) {
        const int ra = p.r[l], rb = p.r[l + 1], R2 = max(ra, rb);
        for (int t = lane; t <= 2 * R2; t += 32) {
            const int ta = t - R2 + ra, tb = t - R2 + rb;
            const bool ia = ta >= 0 && ta <= 2 * ra, ib = tb >= 0 && tb <= 2 * rb;
            p.wt[p.wtoff[l] + t] = make_float4(ia ? p.w[p.woff[l] + ta] : 0.0f, ia ? p.dw[p.woff[l] + ta] : 0.0f,
                                               ib ? p.w[p.woff[l + 1] + tb] : 0.0f,
                                               ib ? p.dw[p.woff[l + 1] + tb] : 0.0f);
        }
    }
}

// What a soft call starts from, in one launch: block 0 clears the counters and
// sums, builds the tap, coefficient and bin-weight tables of the device sigmas
// (skipped when the sigmas equal those the tables were last built from: a batch
// of frames at one ladder builds them once; last_sig is NaN after allocation)
// and folds dloss/dH into one weight per plane; the other blocks empty the
// record path's lists.
__global__ void __launch_bounds__(PREP_THREADS) soft_prep_kernel(const __grid_constant__ SoftPrep p) {
    if (blockIdx.x > 0) {
        const Lists a = frame_lists(p.lists, p.H, p.W, blockIdx.y);
        const int h0 = (blockIdx.x - 1) * PREP_CELLS;
        for (int i = h0 + threadIdx.x; i < min(h0 + PREP_CELLS, 3 * a.n_cells); i += PREP_THREADS)
            a.count[i] = i < 2 * a.n_cells ? 0 : -1;   // count, linked; head
        return;
    }
    if (blockIdx.y > 0) return;
    for (int i = threadIdx.x; i < p.n_zero; i += PREP_THREADS) p.zero[i] = 0;
    for (int i = threadIdx.x; i < p.n_acc; i += PREP_THREADS) p.acc[i] = 0.0;
    bool changed = false;
    for (int i = threadIdx.x; i < p.K; i += blockDim.x) changed |= !(p.sig[i] == p.last_sig[i]);
    if (__syncthreads_or(changed)) soft_tables(p);
    if (p.gH == nullptr) return;
    __syncthreads();
    for (int l = threadIdx.x; l < 2 * p.P; l += PREP_THREADS) {
        const float* kap = l < p.P ? p.kappa + l * p.nbins : p.dkappa + (l - p.P) * p.nbins;
        float a = 0.0f;
#pragma unroll 8
        for (int k = 0; k < p.nbins; ++k) a += p.gH[k] * kap[k];
        p.gk[l] = a;
    }
}
static SoftPrep prep_params(dog_handle* h, SoftWS* ws, const float* sig) {
    const FusedParams& b = handle_base(h);
    const std::vector<double>& ref = handle_sigmas(h);
    SoftPrep q{};
    q.sig = sig;
    q.K = b.K;
    q.P = b.P;
    q.nbins = handle_cfg(h).nbins;
    q.norm = handle_cfg(h).norm;
    for (int i = 0; i < b.K; ++i) {
        q.r[i] = handle_levels(h)[i].r;
        q.woff[i] = handle_levels(h)[i].woff;
        q.tpad[i] = handle_levels(h)[i].tpad;
        handle_tap_slot(h, i, &q.pbase[i], &q.plead[i]);
        q.padoff[i] = pad_offset(h, i);
    }
    q.lref0 = std::log(ref[0]);
    q.lrefP = std::log(ref[b.P - 1]);
    q.w = ws->w;
    q.dw = ws->dw;
    q.wp = ws->wp;
    q.c = ws->c;
    q.kappa = ws->kappa;
    q.dkappa = ws->dkappa;
    q.last_sig = ws->last_sig;
    q.wt = ws->wt;
    q.wpad = ws->wpad;
    q.gk = ws->gk;
    for (int l = 0, n = 0; l < b.P; ++l) {
        q.wtoff[l] = n;
        n += 2 * plane_radius(h, l) + 1;
    }
    return q;
}

static FusedParams soft_fused(dog_handle* h, SoftWS* ws, const float* img, int n, long long stride, int H, int W,
                              int pitch, int mode) {
    FusedParams p = handle_base(h);
    p.img = img;
    p.dtype = DOG_DTYPE_F32;
    p.H = H;
    p.W = W;
    p.pitch = pitch;
    // overlapping strips (32 columns stepping by 30): every local maximum is
    // settled inside the fused kernel, so no strip-edge resolve follows (the
    // soft modes keep every maximum, thousands per frame at strip edges)
    p.overlap = 1;
    p.strip_step = TX - 2;
    p.strip_x0 = -1;
    p.n_strips = (W + TX - 2 - 1) / (TX - 2);
    p.band = pick_band(p, handle_sms(h), H, n * p.n_strips, std::min(handle_band(h), H));
    p.n_bands = (H + p.band - 1) / p.band;
    p.frames = nullptr;
    p.n_frames = n;
    p.frame_stride = stride;
    p.mode = mode;
    p.w = ws->wp;
    p.c = ws->c;
    p.kappa = ws->kappa;
    p.dkappa = ws->dkappa;
    p.nbins = handle_cfg(h).nbins;
    p.inv_T = (float)(1.0 / handle_cfg(h).soft_T);
    p.status = handle_status(h);
    return p;
}

// Frames of a batch whose lists the workspace holds: grown to the batch unless
// the stream is being captured (then the batch goes in several passes).  A graph
// captured earlier keeps the address of the lists of its time, so outgrown ones
// are kept with the workspace; each growth but the last at least doubles the
// frames, so that there are at most seven, together below twice the last.
static int list_frames(SoftWS* ws, int n, cudaStream_t s) {
    const size_t one = sizeof(int) * (size_t)frame_lists(nullptr, ws->H, ws->W, 0).ints;
    const int most = (int)std::max<size_t>(1, std::min((size_t)LIST_FRAMES, LIST_BYTES / one));
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (std::min(n, most) > ws->n_lists && cudaStreamIsCapturing(s, &cap) == cudaSuccess &&
        cap == cudaStreamCaptureStatusNone) {
        const int want = std::min(most, std::max(n, 2 * ws->n_lists));
        void* more = nullptr;
        if (cudaMalloc(&more, want * one) == cudaSuccess) {
            ws->old_lists[ws->n_old++] = ws->lists;
            ws->lists = more;
            ws->n_lists = want;
        } else {
            cudaGetLastError();
        }
    }
    return std::min(n, ws->n_lists);
}

#define SOFT_CUDA(x)                                                                  \
    do {                                                                              \
        cudaError_t e_ = (x);                                                         \
        if (e_ != cudaSuccess) return e_ == cudaErrorMemoryAllocation ? DOG_ERR_NOMEM : DOG_ERR_CUDA; \
    } while (0)

int soft_forward(dog_handle* h, const float* img, int n, long long stride, int H, int W, int pitch, const float* sig,
                 float* out, dog_soft_max* rec, int rec_cap, int* rec_count, cudaStream_t s) {
    SoftWS* ws = nullptr;
    int st = soft_ws(h, H, W, &ws);
    if (st != DOG_OK) return st;
    SoftPrep q = prep_params(h, ws, sig);
    if (rec != nullptr) {
        q.zero = rec_count;
        q.n_zero = n;
    }
    soft_prep_kernel<<<1, PREP_THREADS, 0, s>>>(q);
    SOFT_CUDA(cudaGetLastError());
    FusedParams p = soft_fused(h, ws, img, n, stride, H, W, pitch, MODE_SOFT);
    p.soft_out = out;
    if (rec != nullptr) {
        p.rec = rec;
        p.rec_cap = rec_cap;
        p.rec_count = rec_count;
    }
    SOFT_CUDA(timed_fused(h, p, n * p.n_strips * p.n_bands, s));
    return DOG_OK;
}

// ---------------------------------------------------------------------------
__device__ __forceinline__ int refl_i(int i, int n) {
    if (i >= 0 && i < n) return i;   // inside: no modulo
    int p = 2 * n;
    int m = i % p;
    if (m < 0) m += p;
    return m >= n ? p - 1 - m : m;
}

struct AdjParams {
    float* A;
    float* Y;
    float* Yd;
    const float* img;
    int pitch;
    float* gimg;
    int H, W, K, R;
    const float* w;
    const float* dw;
    int r[MAX_LEVELS];
    int tpad[MAX_LEVELS];
    int woff[MAX_LEVELS];
    double* dw_acc;
};

// Dense adjoints.  Both kernels of a level, w(t) and dw/dsigma(t), are even in t
// and the boundary reflects about the half sample, so the adjoint of a blur is
// the same blur: out(m) = sum_{u < Tpad} k[u] X(refl(m - r + u)) over zero-padded
// taps (cells that only padding taps reach are zero).  Eight consecutive outputs
// per thread are accumulated against a two-window register file (8 inputs per
// block of 8 taps), for two tap sets at once.
__device__ __forceinline__ void tap_block2(float (&o)[8], float (&od)[8], const float (&A)[8], const float (&B)[8],
                                           const float* __restrict__ w, const float* __restrict__ dw) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float a = w[u], b = dw[u];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float x = (k + u < 8) ? A[k + u] : B[k + u - 8];
            o[k] = __fmaf_rn(a, x, o[k]);
            od[k] = __fmaf_rn(b, x, od[k]);
        }
    }
}

// out[k] = sum_u w[u] X[(k + u) st], od[k] with dw; u < 8 nb.
__device__ __forceinline__ void corr8x2(const float* __restrict__ X, int st, const float* __restrict__ w,
                                        const float* __restrict__ dw, int nb, float (&o)[8], float (&od)[8]) {
    float A[8], B[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        o[k] = 0.0f;
        od[k] = 0.0f;
        A[k] = X[k * st];
    }
    int j = 0;
    for (;;) {
#pragma unroll
        for (int k = 0; k < 8; ++k) B[k] = X[(8 * j + 8 + k) * st];
        tap_block2(o, od, A, B, w + 8 * j, dw + 8 * j);
        if (++j == nb) break;
#pragma unroll
        for (int k = 0; k < 8; ++k) A[k] = X[(8 * j + 8 + k) * st];
        tap_block2(o, od, B, A, w + 8 * j, dw + 8 * j);
        if (++j == nb) break;
    }
}

// One tap set: out[k] = sum_u w[u] X[(k + u) st], u < 8 nb.
__device__ __forceinline__ void corr8(const float* __restrict__ X, int st, const float* __restrict__ w, int nb,
                                      float (&o)[8]) {
    float A[8], B[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        o[k] = 0.0f;
        A[k] = X[k * st];
    }
    int j = 0;
    for (;;) {
#pragma unroll
        for (int k = 0; k < 8; ++k) B[k] = X[(8 * j + 8 + k) * st];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int k = 0; k < 8; ++k) o[k] = __fmaf_rn(w[8 * j + u], (k + u < 8) ? A[k + u] : B[k + u - 8], o[k]);
        if (++j == nb) break;
#pragma unroll
        for (int k = 0; k < 8; ++k) A[k] = X[(8 * j + 8 + k) * st];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int k = 0; k < 8; ++k) o[k] = __fmaf_rn(w[8 * j + u], (k + u < 8) ? B[k + u] : A[k + u - 8], o[k]);
        if (++j == nb) break;
    }
}

// Column adjoint of level i, columns x0 .. x0 + 31 and rows m0 .. m0 + 8 WARPS - 1:
// Y_i = B_y^T A_i (kernel w_i) and, when SIG, Yd_i (dw_i) for the sigma
// gradient; warp g on rows 8g .. 8g+7, lane = column.
__host__ __device__ inline int adj_y_smem_floats(int warps, int tpad_max) {
    return (8 * warps + tpad_max + 8) * 32 + 2 * tpad_max;
}
template <bool SIG, int WARPS>
__device__ __forceinline__ void adj_y_tile(const AdjParams& p, float* ysm, int x0, int m0, int i) {
    const int r = p.r[i], tpad = p.tpad[i], nb = tpad >> 3;
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int rows = 8 * WARPS + tpad + 8;
    float* X = ysm;                  // rows x 32: A rows m0 - r + j, reflected
    float* ws = ysm + rows * 32;     // tpad
    float* wd = ws + tpad;           // tpad
    const size_t plane = (size_t)p.H * p.W;
    const float* A = p.A + plane * i;
    for (int t = threadIdx.x; t < tpad; t += 32 * WARPS) {
        ws[t] = p.w[p.woff[i] + t];
        wd[t] = p.dw[p.woff[i] + t];
    }
    const int x = x0 + lane;
    // warp g stages rows g, g + WARPS, ...; eight loads in flight before the stores
    for (int j0 = g; j0 < rows; j0 += 8 * WARPS) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = j0 + WARPS * u, n = m0 - r + j;
            v[u] = (j < rows && n >= -r && n < p.H + r && x < p.W) ? __ldcg(A + (size_t)refl_i(n, p.H) * p.W + x) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j0 + WARPS * u < rows) X[(j0 + WARPS * u) * 32 + lane] = v[u];
    }
    __syncthreads();
    float o[8], od[8];
    if (SIG)
        corr8x2(X + 8 * g * 32 + lane, 32, ws, wd, nb, o, od);
    else
        corr8(X + 8 * g * 32 + lane, 32, ws, nb, o);
    if (x >= p.W) return;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int m = m0 + 8 * g + k;
        if (m >= p.H) break;
        p.Y[plane * i + (size_t)m * p.W + x] = o[k];
        if (SIG) p.Yd[plane * i + (size_t)m * p.W + x] = od[k];
    }
}

constexpr int ADJ_WARPS = 8;
__global__ void __launch_bounds__(32 * ADJ_WARPS) adj_y_kernel(const __grid_constant__ AdjParams p) {
    extern __shared__ float ysm[];
    adj_y_tile<true, ADJ_WARPS>(p, ysm, blockIdx.x * 32, blockIdx.y * 8 * ADJ_WARPS, blockIdx.z);
}

constexpr int ADJ_XR = 32;     // output rows per CTA of the row adjoint (4 warps x 8)

__host__ __device__ inline int adj_x_stride_y(int tpad_max) { return (32 + tpad_max + 8) | 1; }
__host__ __device__ inline int adj_x_stride_i(int R) { return (32 + 2 * R + 16) | 1; }
__host__ __device__ inline int adj_x_smem_floats(int tpad_max, int R, bool sig) {
    return ADJ_XR * (adj_x_stride_y(tpad_max) + (sig ? adj_x_stride_i(R) : 0)) + 2 * tpad_max;
}

// Row adjoint summed over levels into dloss/dI and, when SIG, the kernel-shape part of
// dloss/dsigma_i = <Y_i, B_x' I> + <Yd_i, B_x I>.  128 threads cover 32 columns x 32
// rows; lane (rho, g) of warp q owns row 8q + rho, columns 8g .. 8g+7.
template <bool SIG>
__device__ __forceinline__ void adj_x_tile(const AdjParams& p, float* xsm, double (*red)[MAX_LEVELS], int tpad_max,
                                           int x0, int y0) {
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int rho = lane >> 2, g4 = lane & 3;
    const int row = 8 * q + rho;                 // 0 .. 31
    const int y = y0 + row;
    const int SY = adj_x_stride_y(tpad_max), SI = adj_x_stride_i(p.R);
    float* Yt = xsm;                              // ADJ_XR x SY: Y_i rows, columns x0 - r + c, reflected
    float* It = Yt + ADJ_XR * SY;                 // ADJ_XR x SI: image rows, columns x0 - R + c, reflected
    float* ws = SIG ? It + ADJ_XR * SI : It;      // tpad_max (no image tile without SIG)
    float* wd = ws + tpad_max;                    // tpad_max
    const size_t plane = (size_t)p.H * p.W;
    const int R = p.R;
    // image rows y0 .. y0+31 (clamped), columns x0-R .. x0+R+47 (reflected);
    // thread t stages columns t, t + 128 of every row
    if (SIG) {
        const int c0 = threadIdx.x, c1 = threadIdx.x + 128;
        const int xr0 = refl_i(x0 - R + c0, p.W), xr1 = refl_i(x0 - R + c1, p.W);
        const bool ok0 = c0 < 32 + 2 * R + 16, ok1 = c1 < 32 + 2 * R + 16;
        for (int rr0 = 0; rr0 < ADJ_XR; rr0 += 8) {   // 16 loads in flight before the stores
            float v0[8], v1[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float* src = p.img + (size_t)min(y0 + rr0 + u, p.H - 1) * p.pitch;
                v0[u] = ok0 ? __ldg(src + xr0) : 0.0f;
                v1[u] = ok1 ? __ldg(src + xr1) : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (c0 < SI) It[(rr0 + u) * SI + c0] = v0[u];
                if (c1 < SI) It[(rr0 + u) * SI + c1] = v1[u];
            }
        }
    }
    float gsum[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) gsum[k] = 0.0f;
    for (int i = 0; i < p.K; ++i) {
        const int r = p.r[i], tpad = p.tpad[i], nb = tpad >> 3;
        const float* Yi = p.Y + plane * i;
        const float* Ydi = p.Yd + plane * i;
        __syncthreads();
        for (int t = threadIdx.x; t < tpad; t += blockDim.x) {
            ws[t] = p.w[p.woff[i] + t];
            wd[t] = p.dw[p.woff[i] + t];
        }
        const int wt = 32 + tpad + 8;
        // Y_i rows y0 .. y0+31, columns x0-r .. x0-r+wt-1 (reflected)
        const int xs = x0 - r;
        const int xa = xs >= 0 ? xs & ~3 : -((3 - xs) & ~3);   // xs rounded down to a multiple of 4
        const int off = xs - xa, n4 = (wt + off + 3) >> 2;     // float4 columns per row
        if ((p.W & 3) == 0 && xa >= 0 && xa + 4 * n4 <= p.W && y0 + ADJ_XR <= p.H) {
            // interior tile: 16-byte loads, thread (row phase, float4 column),
            // four rows' loads in flight
            const int rpp = 128 / n4, r0 = threadIdx.x / n4, c4 = threadIdx.x - r0 * n4;
            if (r0 < rpp) {
                const float4* src = reinterpret_cast<const float4*>(Yi + (size_t)y0 * p.W + xa) + c4;
                const int row4 = p.W >> 2;
                for (int rb = r0; rb < ADJ_XR; rb += 4 * rpp) {
                    float4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int rr = min(rb + u * rpp, ADJ_XR - 1);
                        v[u] = __ldcg(src + (size_t)rr * row4);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int rr = rb + u * rpp;
                        if (rr < ADJ_XR) {
                            float* d = Yt + rr * SY + 4 * c4 - off;   // column 4 c4 + k - off of the tile
                            const float e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (4 * c4 + k - off >= 0 && 4 * c4 + k - off < wt) d[k] = e[k];
                        }
                    }
                }
            }
        } else {
            const int c0 = threadIdx.x, c1 = threadIdx.x + 128;
            const int xx0 = xs + c0, xx1 = xs + c1;
            const bool ok0 = c0 < wt && xx0 < p.W + r, ok1 = c1 < wt && xx1 < p.W + r;
            const int xr0 = refl_i(xx0, p.W), xr1 = refl_i(xx1, p.W);
            for (int rr0 = 0; rr0 < ADJ_XR; rr0 += 8) {   // 16 loads in flight before the stores
                float v0[8], v1[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int yy = y0 + rr0 + u;
                    const float* src = Yi + (size_t)yy * p.W;
                    v0[u] = (ok0 && yy < p.H) ? __ldcg(src + xr0) : 0.0f;
                    v1[u] = (ok1 && yy < p.H) ? __ldcg(src + xr1) : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (c0 < wt) Yt[(rr0 + u) * SY + c0] = v0[u];
                    if (c1 < wt) Yt[(rr0 + u) * SY + c1] = v1[u];
                }
            }
        }
        __syncthreads();
        float z[8], hb[8], hd[8];
        corr8(Yt + row * SY + 8 * g4, 1, ws, nb, z);
        if (SIG) corr8x2(It + row * SI + (R - r) + 8 * g4, 1, ws, wd, nb, hb, hd);    // B_x I and B_x' I
        // this thread's 16 products in FP32 (one rounding each, as the inputs
        // are FP32), then the warp's sum in FP64 (the FP64 pipe is slow here)
        float dotf = 0.0f;
        if (y < p.H) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int x = x0 + 8 * g4 + k;
                if (x >= p.W) break;
                gsum[k] += z[k];
                if (SIG) {
                    const float yv = Yt[row * SY + r + 8 * g4 + k];   // Y_i(y, x)
                    dotf = __fmaf_rn(yv, hd[k], __fmaf_rn(Ydi[(size_t)y * p.W + x], hb[k], dotf));
                }
            }
        }
        if (SIG) {
            double dot = (double)dotf;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            if (lane == 0) red[q][i] = dot;
        }
    }
    if (y < p.H) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int x = x0 + 8 * g4 + k;
            if (x < p.W) p.gimg[(size_t)y * p.W + x] = gsum[k];
        }
    }
    if (!SIG) return;
    __syncthreads();
    for (int i = threadIdx.x; i < p.K; i += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < 4; ++w) s += red[w][i];
        if (s != 0.0) atomicAdd(&p.dw_acc[i], s);
    }
}

__global__ void __launch_bounds__(128) adj_x_kernel(const __grid_constant__ AdjParams p, int tpad_max) {
    extern __shared__ float xsm[];
    __shared__ double red[4][MAX_LEVELS];
    adj_x_tile<true>(p, xsm, red, tpad_max, blockIdx.x * 32, blockIdx.y * ADJ_XR);
}

struct FinParams {
    const float* sig;
    int K, P, norm;
    double lref0, lrefP;
    const double* acc;   // dc (P), dt (P), dw (K), ACC_COPIES times
    float* gsig;
};

// dloss/dsigma_i from the sums (accumulated into gsig); thread i on level i.
__device__ __forceinline__ void soft_finalize(const FinParams& p, int i) {
    if (i >= p.K) return;
    double g = 0.0, dc = 0.0, dt = 0.0, dcl = 0.0;   // dw_i, dc_i, dt_i, dc_{i-1}
#pragma unroll
    for (int c = 0; c < ACC_COPIES; ++c) {
        const double* a = p.acc + c * (2 * p.P + p.K);
        g += a[2 * p.P + i];
        if (i < p.P) {
            dc += a[i];
            dt += a[p.P + i];
        }
        if (i > 0) dcl += a[i - 1];
    }
    const double si = (double)p.sig[i];
    if (p.norm == DOG_NORM_PAPER) {
        if (i < p.P) g += dc;
    } else {
        if (i < p.P) {
            const double d = (double)p.sig[i + 1] - si;
            g += dc * (double)p.sig[i + 1] / (d * d);
        }
        if (i > 0) {
            const double d = si - (double)p.sig[i - 1];
            g -= dcl * (double)p.sig[i - 1] / (d * d);
        }
    }
    if (i < p.P) g += dt / (si * (p.lrefP - p.lref0));
    p.gsig[i] += (float)g;
}

__global__ void soft_finalize_kernel(const __grid_constant__ FinParams p) { soft_finalize(p, threadIdx.x); }

// ---- backward from a recorded list of maxima --------------------------------
// A maximum v in plane l has G_v = gk_l q_v, gk_l = sum_b gH_b kappa_b(t_l), and
//   A_l(v) += c_l G_v,  A_{l+1}(v) -= c_l G_v;
//   dloss/dc_l += gk_l qe_v,  dloss/dt_l += s_v sum_b gH_b dkappa_b(t_l);
//   dloss/dsigma_m += A_m(v) (sum (w'_j w_t + w_j w'_t) I(y + j, x + t))
// for m = l, l + 1, over |j|, |t| <= r_m of the reflected image.
//
// One pass over the record, a chunk of records per CTA at a time:
//  A  a thread per record links it into its cell's list for the gather below;
//  B  the window sums of both levels, with lanes on columns: sum_j w_j I and
//     sum_j w'_j I down the column (four FMAs per pixel for both levels), the
//     column's own weights once at the end.  Windows up to 2 NARROW_R + 1 wide
//     (nearly all: the finest planes) take eight lanes of two columns, wider
//     ones a warp, and those wider than a warp (few: the coarse planes) all the
//     CTA's warps, so that none runs a long serial window;
//  C  the products with G_v, gk and gdk in FP64, lane = record, summed over the
//     lanes of a level (the FP64 pipe takes a warp at two lanes a clock: one
//     record per instruction would bound the kernel).
// A CTA's records are gridDim apart, which evens out the planes.
//
// 16 frames of 1024 x 1024 with 35,000 maxima each, 12 levels, in us: this pass
// 222 (latency of the small windows' loads and the meetings between A, B and C;
// with chunks of 64 records, and so four times the meetings, 277), where a warp
// per maximum with all taps formed per pixel took 830, and its scatter into
// zeroed planes 470.
struct RecParams {
    const dog_soft_max* rec;
    const int* count;
    int cap;
    const float* gk;        // P, then P of dkappa
    const float* c;
    const float4* wt;
    const float* img;
    long long img_stride, rec_stride;   // from a frame to the next
    int pitch;
    int P, K, H, W;
    int r[MAX_LEVELS];
    int wtoff[MAX_LEVELS];
    double* acc;            // dc (P), dt (P), dw (K), ACC_COPIES times
    void* lists;
    FrameFlags* flags;
    int* status;
};

constexpr int REC_WARPS = 8, REC_CHUNK = 256;

// Column sums of a plane's window around (x, y) at offset t - R2: rows j0,
// j0 + j_step, ... of both levels, COLS columns (t, t + 1, ...) at once.  A pixel
// outside a level's own window does not enter its sums.
template <int COLS>
__device__ __forceinline__ void window_sums(const RecParams& p, const float* img, int x, int y, int l, int t, int j0,
                                            int j_step, float& pa, float& pb) {
    const int ra = p.r[l], rb = p.r[l + 1], R2 = max(ra, rb), n2 = 2 * R2 + 1;
    const float4* T = p.wt + p.wtoff[l];
    const bool rows_in = y >= R2 && y + R2 < p.H;
    const float* col[COLS];
#pragma unroll
    for (int c = 0; c < COLS; ++c) col[c] = img + refl_i(x + min(t + c, n2 - 1) - R2, p.W);
    float a0[COLS], a1[COLS], b0[COLS], b1[COLS];
#pragma unroll
    for (int c = 0; c < COLS; ++c) a0[c] = a1[c] = b0[c] = b1[c] = 0.0f;
    for (int jb = j0; jb < n2; jb += 4 * j_step) {
        float px[4][COLS];
        float4 w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = min(jb + u * j_step, n2 - 1), n = y - R2 + j;
            const size_t row = (size_t)(rows_in ? n : refl_i(n, p.H)) * p.pitch;
            w[u] = __ldg(T + j);
#pragma unroll
            for (int c = 0; c < COLS; ++c) px[u][c] = __ldg(col[c] + row);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = jb + u * j_step;
            if (j < n2 && abs(j - R2) <= ra) {
#pragma unroll
                for (int c = 0; c < COLS; ++c) {
                    a0[c] = __fmaf_rn(w[u].x, px[u][c], a0[c]);
                    a1[c] = __fmaf_rn(w[u].y, px[u][c], a1[c]);
                }
            }
            if (j < n2 && abs(j - R2) <= rb) {
#pragma unroll
                for (int c = 0; c < COLS; ++c) {
                    b0[c] = __fmaf_rn(w[u].z, px[u][c], b0[c]);
                    b1[c] = __fmaf_rn(w[u].w, px[u][c], b1[c]);
                }
            }
        }
    }
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
        const float4 w = __ldg(T + min(t + c, n2 - 1));
        if (t + c < n2 && abs(t + c - R2) <= ra) pa = __fmaf_rn(w.y, a0[c], __fmaf_rn(w.x, a1[c], pa));
        if (t + c < n2 && abs(t + c - R2) <= rb) pb = __fmaf_rn(w.w, b0[c], __fmaf_rn(w.z, b1[c], pb));
    }
}

template <int LANES>
__device__ __forceinline__ void sum_lanes(float& a, float& b) {
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
}

__global__ void __launch_bounds__(32 * REC_WARPS) soft_rec_kernel(const __grid_constant__ RecParams p) {
    __shared__ double acc[3 * MAX_LEVELS];
    __shared__ dog_soft_max rec[REC_CHUNK];
    __shared__ float pa[REC_WARPS][REC_CHUNK], pb[REC_WARPS][REC_CHUNK];   // window sums (row 0: of one warp or group)
    __shared__ unsigned char list[3][REC_CHUNK];
    __shared__ int n_list[3];   // narrow, middle, wide windows
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_acc = 2 * p.P + p.K;
    for (int k = tid; k < n_acc; k += blockDim.x) acc[k] = 0.0;
    const int f = blockIdx.y, n = p.count[f];
    const float* img = p.img + f * p.img_stride;
    const dog_soft_max* src = p.rec + f * p.rec_stride;
    const Lists lists = frame_lists(p.lists, p.H, p.W, f);
    const int cells_x = cells(p.W);
    if (n > p.cap && blockIdx.x == 0 && tid == 0) atomicCAS(p.status, 0, (int)DOG_ERR_CAPACITY);
    const int m = min(n, p.cap);
    const long long step = gridDim.x;
    for (long long c0 = blockIdx.x; c0 < m; c0 += step * REC_CHUNK) {
        const int here = (int)min((m - c0 + step - 1) / step, (long long)REC_CHUNK);
        __syncthreads();
        if (tid < 3) n_list[tid] = 0;
        __syncthreads();
        if (tid < here) {
            const long long i = c0 + tid * step;
            dog_soft_max v = src[i];
            const int l = v.level;
            if (v.x < 0 || v.x >= p.W || v.y < 0 || v.y >= p.H || l < 0 || l >= p.P) {   // not this frame's record
                atomicCAS(p.status, 0, (int)DOG_ERR_INVALID);
                rec[tid].level = -1;
            } else {
                const float G = __ldg(p.c + l) * (__ldg(p.gk + l) * v.q);
                const int R2 = max(p.r[l], p.r[l + 1]);
                const int which = R2 <= NARROW_R ? 0 : R2 < 16 ? 1 : 2;
                list[which][atomicAdd(&n_list[which], 1)] = (unsigned char)tid;
                if (!(G == 0.0f)) {
                    const int cell = (v.y >> CELL_SHIFT) * cells_x + (v.x >> CELL_SHIFT);
                    int4 e = make_int4(v.x, v.y * 32 + l, __float_as_int(G), 0);
                    const int at = which == 0 ? atomicAdd(lists.count + cell, 1) : CELL_SLOTS;
                    if (at < CELL_SLOTS) {
                        lists.slots[(long long)cell * CELL_SLOTS + at] = e;
                    } else {
                        const int k = atomicAdd(&p.flags[f].linked, 1);
                        if (k >= lists.ent_cap || atomicAdd(lists.linked + cell, 1) >= CHAIN_MAX) {
                            p.flags[f].dense = 1;
                        } else {
                            e.w = atomicExch(lists.head + cell, k);
                            lists.ent[k] = e;
                        }
                    }
                }
                v.q = G;
                rec[tid] = v;
            }
        }
        __syncthreads();
        const int n_narrow = n_list[0], n_mid = n_list[1], n_wide = n_list[2];
        for (int k0 = 4 * warp; k0 < n_narrow; k0 += 4 * REC_WARPS) {
            const int k = list[0][min(k0 + (lane >> 3), n_narrow - 1)];
            float a = 0.0f, b = 0.0f;
            window_sums<2>(p, img, rec[k].x, rec[k].y, rec[k].level, 2 * (lane & 7), 0, 1, a, b);
            sum_lanes<8>(a, b);
            if ((lane & 7) == 0 && k0 + (lane >> 3) < n_narrow) { pa[0][k] = a; pb[0][k] = b; }
        }
        for (int q = warp; q < n_mid; q += REC_WARPS) {
            const int k = list[1][q];
            float a = 0.0f, b = 0.0f;
            window_sums<1>(p, img, rec[k].x, rec[k].y, rec[k].level, lane, 0, 1, a, b);
            sum_lanes<32>(a, b);
            if (lane == 0) { pa[0][k] = a; pb[0][k] = b; }
        }
        for (int q = 0; q < n_wide; ++q) {
            const int k = list[2][q], l = rec[k].level, n2 = 2 * max(p.r[l], p.r[l + 1]) + 1;
            float a = 0.0f, b = 0.0f;
            for (int t = lane; t < n2; t += 32) window_sums<1>(p, img, rec[k].x, rec[k].y, l, t, warp, REC_WARPS, a, b);
            sum_lanes<32>(a, b);
            if (lane == 0) { pa[warp][k] = a; pb[warp][k] = b; }
        }
        __syncthreads();
        if (warp < REC_CHUNK / 32) {
            const int k = 32 * warp + lane, l = k < here ? rec[k].level : -1;
            double v[4] = {0.0, 0.0, 0.0, 0.0};
            if (l >= 0) {
                const double G = (double)rec[k].q;
                v[0] = G * (double)pa[0][k];
                v[1] = -G * (double)pb[0][k];
                if (max(p.r[l], p.r[l + 1]) >= 16)
                    for (int w = 1; w < REC_WARPS; ++w) {
                        v[0] += G * (double)pa[w][k];
                        v[1] -= G * (double)pb[w][k];
                    }
                v[2] = (double)__ldg(p.gk + l) * (double)rec[k].qe;
                v[3] = (double)rec[k].s * (double)__ldg(p.gk + p.P + l);
            }
            for (unsigned left = __ballot_sync(0xffffffffu, l >= 0); left;) {
                const int lv = __shfl_sync(0xffffffffu, l, __ffs(left) - 1);
                const unsigned same = __ballot_sync(0xffffffffu, l == lv);
                left &= ~same;
                const int to[4] = {2 * p.P + lv, 2 * p.P + lv + 1, lv, p.P + lv};
                if (__popc(same) <= 3) {
                    if (l == lv)
                        for (int f = 0; f < 4; ++f) atomicAdd(&acc[to[f]], v[f]);
                    continue;
                }
#pragma unroll
                for (int f = 0; f < 4; ++f) {
                    double t = l == lv ? v[f] : 0.0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                    if (lane == f) atomicAdd(&acc[to[f]], t);
                }
            }
        }
    }
    __syncthreads();
    for (int k = tid; k < n_acc; k += blockDim.x)
        if (acc[k] != 0.0) atomicAdd(p.acc + (blockIdx.x % ACC_COPIES) * n_acc + k, acc[k]);
}

// dloss/dI of a 32 x 32 tile from the lists.  B_i is symmetric, so pixel m gets
//   sum over maxima v of plane A_i of A_i(v) w_i(m_y - v_y) w_i(m_x - v_x),
// v running over the maxima and their mirror images in the frame's edges.
// The CTA walks the cells around the tile (those of narrow planes only nearby),
// keeps the (maximum, level) pairs whose windows reach the tile, orders them by
// level and place (so that the sum does not depend on the lists' order), and
// each warp adds its pairs to 8 rows, lane = column.  A tile that more than
// TILE_PAIRS pairs reach asks for the frame's dense form.
//
// The planes are nearly empty (three maxima in a hundred voxels of the finest,
// one in a thousand of the next): about 116 pairs reach a tile, where blurring
// the planes is 900 multiply-adds a pixel.  16 frames of 1024 x 1024, 12 levels:
// 260 us, where the two dense passes and their edge folds took 2260.
struct TileParams {
    void* lists;
    FrameFlags* flags;
    int H, W, K, R;
    const float* wpad;      // all levels' taps, TAP_PAD zeros around each
    int r[MAX_LEVELS];
    int soff[MAX_LEVELS];   // level's taps in wpad
    int n_taps;
    float* gimg;
};

constexpr int TILE = 32, TILE_WARPS = 4, TILE_ROWS = TILE / TILE_WARPS, TILE_PAIRS = 512;
constexpr int NEAR = (TILE >> CELL_SHIFT) + 2;   // cells per side within NARROW_R of a tile
static_assert(NARROW_R <= 1 << CELL_SHIFT, "narrow planes reach one cell beyond a tile");

// Shared memory: the pairs, then the taps twice, the second time one float on
// (so that two rows' taps are one aligned load at either parity).
constexpr int PAIR_BYTES = TILE_PAIRS * (int)(sizeof(int4) + sizeof(unsigned) + sizeof(int2));
static __host__ __device__ int tap_copy(int n_taps) { return (n_taps + 3) & ~1; }   // floats of a copy
constexpr int TILE_SMEM_MAX =
    PAIR_BYTES + (int)sizeof(float) * 2 * (TAP_PAD + MAX_LEVELS * (2 * DOG_MAX_RADIUS + 1 + TAP_PAD) + 4);

__global__ void __launch_bounds__(32 * TILE_WARPS) soft_tile_kernel(const __grid_constant__ TileParams p) {
    extern __shared__ __align__(16) unsigned char tsm[];
    __shared__ int n_pairs;
    // sorted: first and last of the tile's rows in the window; byte offsets of
    // column 0's tap, of row 0's tap (in the copy where it is 8-byte aligned); A
    int4* sorted = reinterpret_cast<int4*>(tsm);
    unsigned* keys = reinterpret_cast<unsigned*>(sorted + TILE_PAIRS);   // level, sign, y, x, place in `found`
    int2* found = reinterpret_cast<int2*>(keys + TILE_PAIRS);            // level's taps | r << 16, A
    float* taps = reinterpret_cast<float*>(tsm + PAIR_BYTES);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x0 = blockIdx.x * TILE, y0 = blockIdx.y * TILE, frame = blockIdx.z;
    if (p.flags[frame].dense) return;   // (this launch does not write it)
    const Lists lists = frame_lists(p.lists, p.H, p.W, frame);
    const int cells_x = cells(p.W), cells_y = cells(p.H);
    // nearby cells' counts, and the heads of all cells within R: one lane per
    // cell of a row of cells (at most 21), a row per warp
    constexpr int NU = (NEAR * NEAR * CELL_SLOTS + 32 * TILE_WARPS - 1) / (32 * TILE_WARPS);
    int4 slot[NU];
    {
        const int4* at[NU];
        bool has[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) {   // slot by slot, so that a warp's lanes are of one fullness
            const int k = tid + 32 * TILE_WARPS * u, s = k / (NEAR * NEAR), c = k % (NEAR * NEAR);
            const int cx = (x0 >> CELL_SHIFT) - 1 + c % NEAR, cy = (y0 >> CELL_SHIFT) - 1 + c / NEAR;
            const bool in = s < CELL_SLOTS && cx >= 0 && cx < cells_x && cy >= 0 && cy < cells_y;
            const int cell = in ? cy * cells_x + cx : 0;
            has[u] = in && s < __ldg(lists.count + cell);
            at[u] = lists.slots + (long long)cell * CELL_SLOTS + s;
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) slot[u] = has[u] ? __ldg(at[u]) : make_int4(0, 0, 0, -1);
    }
    if (tid == 0) n_pairs = 0;
    const int copy = tap_copy(p.n_taps);
#pragma unroll 8
    for (int t = tid; t < p.n_taps; t += 32 * TILE_WARPS) taps[t] = taps[copy + t + 1] = __ldg(p.wpad + t);
    if (tid == 0) taps[copy] = 0.0f;
    __syncthreads();
    auto keep = [&](const int4& v) {   // the pairs of a maximum with its two levels
        const int l = v.y & 31, vx = v.x, vy = v.y >> 5;
#pragma unroll 1
        for (int s = 0; s < 2; ++s) {
            const int i = l + s, r = p.r[i];
            // a mirror image is never nearer to a pixel of the frame than the maximum itself
            if (vx + r < x0 || vx - r >= x0 + TILE || vy + r < y0 || vy - r >= y0 + TILE) continue;
            // images k N + (k odd ? N - 1 - v : v) in the edges of a line of N
            const int kx = vx >= r && vx + r < p.W ? 0 : (r + p.W - 1) / p.W;
            const int ky = vy >= r && vy + r < p.H ? 0 : (r + p.H - 1) / p.H;
            for (int a = -ky; a <= ky; ++a) {
                const int y = a * p.H + (a & 1 ? p.H - 1 - vy : vy);
                if (y + r < y0 || y - r >= y0 + TILE) continue;
                for (int b = -kx; b <= kx; ++b) {
                    const int x = b * p.W + (b & 1 ? p.W - 1 - vx : vx);
                    if (x + r < x0 || x - r >= x0 + TILE) continue;
                    const int at = atomicAdd(&n_pairs, 1);
                    if (at >= TILE_PAIRS) continue;
                    keys[at] = (unsigned)(2 * i + s) << 26 | (y - y0 + DOG_MAX_RADIUS) << 18 |
                               (x - x0 + DOG_MAX_RADIUS) << 10 | at;
                    found[at] = make_int2(p.soff[i] | r << 16, s ? v.z ^ (int)0x80000000 : v.z);
                }
            }
        }
    };
#pragma unroll
    for (int u = 0; u < NU; ++u)
        if (slot[u].w == 0) keep(slot[u]);
    {
        const int cxa = max(x0 - p.R, 0) >> CELL_SHIFT, cxb = min((x0 + TILE - 1 + p.R) >> CELL_SHIFT, cells_x - 1);
        const int cya = max(y0 - p.R, 0) >> CELL_SHIFT, cyb = min((y0 + TILE - 1 + p.R) >> CELL_SHIFT, cells_y - 1);
        const int cx = cxa + lane;
        for (int cy0 = cya + warp; cy0 <= cyb; cy0 += 4 * TILE_WARPS) {
            int e[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int cy = cy0 + u * TILE_WARPS;
                e[u] = cy <= cyb && cx <= cxb ? __ldg(lists.head + cy * cells_x + cx) : -1;
            }
            while (e[0] >= 0 || e[1] >= 0 || e[2] >= 0 || e[3] >= 0) {   // the four lists side by side
                int4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e[u] >= 0) v[u] = __ldg(lists.ent + e[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (e[u] >= 0) {
                        e[u] = v[u].w;
                        keep(v[u]);
                    }
            }
        }
    }
    __syncthreads();
    const int n = n_pairs;
    if (n > TILE_PAIRS) {
        if (tid == 0) p.flags[frame].tiles = 1;
        return;
    }
    const int n4 = (n + 3) >> 2;
    if (tid < 4 * n4 - n) keys[n + tid] = 0xffffffffu;
    __syncthreads();
    for (int k = tid; k < n; k += 32 * TILE_WARPS) {
        const unsigned key = keys[k];
        int rank = 0;
#pragma unroll 4
        for (int q = 0; q < n4; ++q) {
            const uint4 o = reinterpret_cast<const uint4*>(keys)[q];
            rank += (o.x < key) + (o.y < key) + (o.z < key) + (o.w < key);
        }
        const int2 f = found[k];
        const int r = f.x >> 16, y = (int)(key >> 18 & 255) - DOG_MAX_RADIUS;
        const int tx = (f.x & 0xffff) + r - (int)(key >> 10 & 255) + DOG_MAX_RADIUS, ty = (f.x & 0xffff) + r - y;
        sorted[rank] = make_int4((y - r) * 65536 + ((y + r) & 0xffff), 4 * tx, 4 * (ty & 1 ? copy + 1 + ty : ty), f.y);
    }
    __syncthreads();
    const int x = x0 + lane, row0 = warp * TILE_ROWS;
    float2 g2[TILE_ROWS / 2];
#pragma unroll
    for (int k = 0; k < TILE_ROWS / 2; ++k) g2[k] = make_float2(0.0f, 0.0f);
    const char* tap_x = reinterpret_cast<const char*>(taps + lane);
    const char* tap_y = reinterpret_cast<const char*>(taps + row0);
    for (int base = 0; base < n; base += 32) {
        bool hit = false;
        if (base + lane < n) {
            const int rows = sorted[base + lane].x;
            hit = (int)(short)(rows & 0xffff) >= row0 && (rows >> 16) < row0 + TILE_ROWS;
        }
        unsigned todo = __ballot_sync(0xffffffffu, hit);
        if (!todo) continue;
        int4 next = sorted[base + __ffs(todo) - 1];
        do {
            const int4 v = next;
            todo &= todo - 1;
            if (todo) next = sorted[base + __ffs(todo) - 1];
            // columns and rows outside the window meet the zeros around the taps
            const float ax = __int_as_float(v.w) * *reinterpret_cast<const float*>(tap_x + v.y);
            const float2 ax2 = make_float2(ax, ax);
            const float2* wy = reinterpret_cast<const float2*>(tap_y + v.z);
#pragma unroll
            for (int k = 0; k < TILE_ROWS / 2; ++k) g2[k] = __ffma2_rn(ax2, wy[k], g2[k]);
        } while (todo);
    }
    if (x >= p.W) return;
    float* out = p.gimg + (size_t)frame * p.H * p.W + (size_t)(y0 + row0) * p.W + x;
#pragma unroll
    for (int k = 0; k < TILE_ROWS; ++k)
        if (y0 + row0 + k < p.H) out[(size_t)k * p.W] = k & 1 ? g2[k >> 1].y : g2[k >> 1].x;
}

// The dense form, for frames whose lists did not do (plateaus, where every voxel
// ties): A cleared, scattered from the record and blurred by the dense passes,
// the grid meeting between them.  One cooperative launch looks after all frames
// of a call, and costs two microseconds when none asks for it.  Block 0 also
// finishes the sigma gradient.
struct DenseParams {
    AdjParams a;
    const dog_soft_max* rec;
    const int* count;
    long long rec_stride;
    int cap, n, P;
    const float* gk;
    const float* c;
    const FrameFlags* flags;
    int* arrived;
    int* status;
    int wait_max;   // rounds of a wait
    int tpad_max;
    FinParams fin;
};

constexpr int DENSE_WARPS = 4;
constexpr int GRID_WAIT_MAX = 1 << 24;   // rounds of a wait, a second or more; then an error

__device__ __forceinline__ bool grid_meet(const DenseParams& p, int target) {
    __shared__ bool met;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(p.arrived, 1);
        met = atomicAdd(p.arrived, 0) >= target;
        for (int spins = 0; !met && spins < p.wait_max; ++spins) {
            __nanosleep(64);
            met = atomicAdd(p.arrived, 0) >= target;
        }
        if (!met) atomicCAS(p.status, 0, (int)DOG_ERR_TIMEOUT);
        __threadfence();
    }
    __syncthreads();
    return met;
}

// What a CTA whose wait ran out leaves in its share of the frames from f on that
// wanted the dense form: no half-made gradient.
__device__ __noinline__ void dense_give_up(const DenseParams& p, int f) {
    const size_t plane = (size_t)p.a.H * p.a.W;
    for (; f < p.n; ++f)
        if (p.flags[f].dense | p.flags[f].tiles)
            for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < plane; k += (size_t)gridDim.x * blockDim.x)
                p.a.gimg[f * plane + k] = __int_as_float(0x7fffffff);
}

__global__ void __launch_bounds__(32 * DENSE_WARPS) soft_dense_kernel(const __grid_constant__ DenseParams p) {
    extern __shared__ float dsm[];
    if (blockIdx.x == 0 && p.fin.gsig != nullptr) soft_finalize(p.fin, threadIdx.x);
    const int grid = gridDim.x;
    int target = 0;
    for (int f = 0; f < p.n; ++f) {
        if (!(p.flags[f].dense | p.flags[f].tiles)) continue;
        AdjParams a = p.a;
        const size_t plane = (size_t)a.H * a.W, first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
        const size_t step = (size_t)grid * blockDim.x;
        a.gimg += f * plane;
        for (size_t k = first; k < plane * a.K; k += step) a.A[k] = 0.0f;
        if (!grid_meet(p, target += grid)) return dense_give_up(p, f);
        const int m = min(p.count[f], p.cap);
        for (long long k = first; k < m; k += step) {
            const dog_soft_max v = p.rec[f * p.rec_stride + k];
            const int l = v.level;
            if (v.x < 0 || v.x >= a.W || v.y < 0 || v.y >= a.H || l < 0 || l >= p.P) continue;   // reported already
            const float G = p.c[l] * (p.gk[l] * v.q);
            float* at = a.A + plane * l + (size_t)v.y * a.W + v.x;
            atomicAdd(at, G);
            atomicAdd(at + plane, -G);
        }
        if (!grid_meet(p, target += grid)) return dense_give_up(p, f);
        const int tx = (a.W + 31) / 32, ty = (a.H + 8 * DENSE_WARPS - 1) / (8 * DENSE_WARPS);
        for (int t = blockIdx.x; t < tx * ty * a.K; t += grid) {
            __syncthreads();
            adj_y_tile<false, DENSE_WARPS>(a, dsm, t % tx * 32, t / tx % ty * 8 * DENSE_WARPS, t / tx / ty);
        }
        if (!grid_meet(p, target += grid)) return dense_give_up(p, f);
        const int tr = (a.H + ADJ_XR - 1) / ADJ_XR;
        for (int t = blockIdx.x; t < tx * tr; t += grid) {
            __syncthreads();
            adj_x_tile<false>(a, dsm, nullptr, p.tpad_max, t % tx * 32, t / tx * ADJ_XR);
        }
        if (!grid_meet(p, target += grid)) return dense_give_up(p, f);
    }
}

static FinParams fin_params(dog_handle* h, SoftWS* ws, const SoftPrep& q, const float* sig, float* gsig) {
    FinParams f{};
    f.sig = sig;
    f.K = q.K;
    f.P = q.P;
    f.norm = handle_cfg(h).norm;
    f.lref0 = q.lref0;
    f.lrefP = q.lrefP;
    f.acc = ws->acc;
    f.gsig = gsig;
    return f;
}

static AdjParams adj_params(dog_handle* h, SoftWS* ws, const float* img, int H, int W, int pitch, float* gimg,
                            int* tpad_max) {
    AdjParams a{};
    a.A = ws->A;
    a.Y = ws->Y;
    a.Yd = ws->Yd;
    a.img = img;
    a.pitch = pitch;
    a.gimg = gimg;
    a.H = H;
    a.W = W;
    a.K = handle_K(h);
    a.w = ws->w;
    a.dw = ws->dw;
    *tpad_max = 8;
    for (int i = 0; i < a.K; ++i) {
        a.r[i] = handle_levels(h)[i].r;
        a.tpad[i] = handle_levels(h)[i].tpad;
        a.woff[i] = handle_levels(h)[i].woff;
        *tpad_max = std::max(*tpad_max, a.tpad[i]);
    }
    a.R = handle_base(h).R;
    a.dw_acc = ws->acc + 2 * handle_P(h);
    return a;
}

int soft_backward(dog_handle* h, const float* img, int H, int W, int pitch, const float* sig,
                  const float* gH, float* gimg, float* gsig, cudaStream_t s) {
    SoftWS* ws = nullptr;
    int st = soft_ws(h, H, W, &ws);
    if (st != DOG_OK) return st;
    const FusedParams& b = handle_base(h);
    const int K = b.K, P = b.P;
    SoftPrep q = prep_params(h, ws, sig);
    q.acc = ws->acc;
    q.n_acc = ACC_COPIES * (2 * P + K);
    soft_prep_kernel<<<1, PREP_THREADS, 0, s>>>(q);
    SOFT_CUDA(cudaGetLastError());
    FusedParams p = soft_fused(h, ws, img, 1, 0, H, W, pitch, MODE_BWD);
    p.gH = gH;
    p.A = ws->A;
    p.dc_acc = ws->acc;
    p.dt_acc = ws->acc + P;
    SOFT_CUDA(timed_fused(h, p, p.n_strips * p.n_bands, s));
    int tpad_max = 0;
    const AdjParams a = adj_params(h, ws, img, H, W, pitch, gimg, &tpad_max);
    dim3 gy((W + 31) / 32, (H + 8 * ADJ_WARPS - 1) / (8 * ADJ_WARPS), K);
    dim3 gx((W + 31) / 32, (H + ADJ_XR - 1) / ADJ_XR);
    adj_y_kernel<<<gy, 32 * ADJ_WARPS, sizeof(float) * adj_y_smem_floats(ADJ_WARPS, tpad_max), s>>>(a);
    SOFT_CUDA(cudaGetLastError());
    adj_x_kernel<<<gx, 128, sizeof(float) * adj_x_smem_floats(tpad_max, b.R, true), s>>>(a, tpad_max);
    SOFT_CUDA(cudaGetLastError());
    soft_finalize_kernel<<<1, MAX_LEVELS, 0, s>>>(fin_params(h, ws, q, sig, gsig));
    SOFT_CUDA(cudaGetLastError());
    return DOG_OK;
}

int soft_backward_rec(dog_handle* h, const float* img, int n, long long stride, int H, int W, int pitch,
                      const float* sig, const dog_soft_max* rec, const int* rec_count, int rec_cap, const float* gH,
                      float* gimg, float* gsig, cudaStream_t s) {
    SoftWS* ws = nullptr;
    int st = soft_ws(h, H, W, &ws);
    if (st != DOG_OK) return st;
    const int K = handle_K(h), P = handle_P(h), sms = handle_sms(h);
    const int per = list_frames(ws, n, s);
    const int n_cells = cells(H) * cells(W);
    FrameFlags* flags = reinterpret_cast<FrameFlags*>(ws->flags);
    int* arrived = reinterpret_cast<int*>(flags + LIST_FRAMES);
    SoftPrep q = prep_params(h, ws, sig);
    q.gH = gH;
    q.zero = ws->flags;
    q.n_zero = (int)(sizeof(FrameFlags) / sizeof(int)) * LIST_FRAMES + 1;
    q.acc = ws->acc;
    q.n_acc = ACC_COPIES * (2 * P + K);
    q.lists = ws->lists;
    q.H = H;
    q.W = W;
    RecParams c{};
    c.cap = rec_cap;
    c.gk = ws->gk;
    c.c = ws->c;
    c.wt = ws->wt;
    c.img_stride = stride;
    c.rec_stride = rec_cap;
    c.pitch = pitch;
    c.P = P;
    c.K = K;
    c.H = H;
    c.W = W;
    c.acc = ws->acc;
    c.lists = ws->lists;
    c.flags = flags;
    c.status = handle_status(h);
    TileParams t{};
    t.lists = ws->lists;
    t.flags = flags;
    t.H = H;
    t.W = W;
    t.K = K;
    t.R = handle_base(h).R;
    t.wpad = ws->wpad;
    t.n_taps = pad_offset(h, K);
    for (int i = 0; i < K; ++i) {
        t.r[i] = c.r[i] = handle_levels(h)[i].r;
        t.soff[i] = q.padoff[i];
        c.wtoff[i] = q.wtoff[i];
    }
    const size_t tile_smem = PAIR_BYTES + sizeof(float) * 2 * tap_copy(t.n_taps);
    if (tile_smem > 48 * 1024)   // the largest any handle needs: other threads may be setting it too
        SOFT_CUDA(cudaFuncSetAttribute(soft_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_SMEM_MAX));
    DenseParams d{};
    d.a = adj_params(h, ws, img, H, W, pitch, gimg, &d.tpad_max);
    d.rec_stride = rec_cap;
    d.cap = rec_cap;
    d.P = P;
    d.gk = ws->gk;
    d.c = ws->c;
    d.flags = flags;
    d.arrived = arrived;
    d.status = handle_status(h);
    d.wait_max = handle_wait_limit(h) < 0 ? GRID_WAIT_MAX : handle_wait_limit(h);
    const size_t dense_smem = sizeof(float) * std::max(adj_y_smem_floats(DENSE_WARPS, d.tpad_max),
                                                       adj_x_smem_floats(d.tpad_max, t.R, false));
    if (ws->dense_grid == 0) {
        int fit = 0;
        SOFT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, soft_dense_kernel, 32 * DENSE_WARPS, dense_smem));
        if (fit < 1) return DOG_ERR_CUDA;
        ws->dense_grid = std::min(fit, 4) * sms;
    }
    for (int first = 0; first < n; first += per) {
        const int now = std::min(per, n - first);
        q.n_lists = now;
        if (first > 0) q.n_acc = 0;
        const dim3 prep_grid(1 + (3 * n_cells + PREP_CELLS - 1) / PREP_CELLS, now);
        soft_prep_kernel<<<prep_grid, PREP_THREADS, 0, s>>>(q);
        SOFT_CUDA(cudaGetLastError());
        c.rec = d.rec = rec + (size_t)first * rec_cap;
        c.count = d.count = rec_count + first;
        c.img = img + first * stride;
        soft_rec_kernel<<<dim3(std::max(1, std::min(rec_cap, 4 * sms / now)), now), 32 * REC_WARPS, 0, s>>>(c);
        SOFT_CUDA(cudaGetLastError());
        t.gimg = d.a.gimg = gimg + (size_t)first * H * W;
        soft_tile_kernel<<<dim3((W + TILE - 1) / TILE, (H + TILE - 1) / TILE, now), 32 * TILE_WARPS, tile_smem, s>>>(t);
        SOFT_CUDA(cudaGetLastError());
        d.n = now;
        if (first + now == n) d.fin = fin_params(h, ws, q, sig, gsig);
        void* args[] = {&d};
        SOFT_CUDA(cudaLaunchCooperativeKernel(soft_dense_kernel, dim3(ws->dense_grid), dim3(32 * DENSE_WARPS), args,
                                              dense_smem, s));
    }
    return DOG_OK;
}

}  // namespace dogk

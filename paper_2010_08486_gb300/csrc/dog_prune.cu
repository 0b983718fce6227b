// Overlap pruning (Sec. 4.1) and blob-volume histogram (Sec. 4) on sm_103a.
//
// Pruning.  The paper coalesces blobs whose normalised overlap exceeds a
// threshold.  Read as a greedy pass in priority order (response descending,
// then level, y, x), a candidate is accepted iff no accepted candidate of
// higher priority conflicts with it; a rejected candidate joins the
// highest-priority accepted candidate it conflicts with.  That outcome is the
// lexicographically-first maximal independent set of the conflict graph in
// priority order, which this kernel computes in parallel rounds: a candidate
// becomes IN once every higher-priority neighbour is OUT, and OUT once any is
// IN.  Round count is bounded by the candidate count (each round settles at
// least the highest-priority undecided candidate).
//
// Conflict test.  Centres are integer pixels, so the squared distance d2 is an
// integer; for a pair of planes (a, b) the host precomputes the smallest
// integer d2 at which the double-precision overlap drops to the threshold
// (overlap decreases with distance).  Two candidates conflict iff
// d2 < d2thr[a][b] -- the device evaluates no transcendental function.
// Neighbours are found through a hashed grid with cells of edge >= the
// largest conflict distance, so all conflicts lie in the 3x3 adjacent cells.
#include <cuda_runtime.h>

#include <atomic>
#include <climits>

#include "dog_internal.cuh"

namespace dogk {

// Histogram bin of one blob (Sec. 4): a blob whose stored sigma equals its
// plane's single-precision sigma takes its plane's precomputed bin; another
// sigma (a coalesced mean) is binned by log volume (LOGV) or by the nearest
// ladder radius in log space (LADDER).
__device__ __forceinline__ int hist_bin(const dog_blob& b, const HistParams& p, const float* sig_f,
                                        const int* level_bin) {
    const int l = min(max(b.level, 0), p.P - 1);
    if (b.sigma == sig_f[l]) return level_bin[l];
    if (p.mode == DOG_HIST_LADDER) {
        const double ls = log((double)b.sigma);
        int best = 0;
        double bd = fabs(ls - p.log_sig[0]);
        for (int q = 1; q < p.P; ++q) {
            const double d = fabs(ls - p.log_sig[q]);
            if (d < bd) { bd = d; best = q; }
        }
        return best;
    }
    const double span = p.log_hi - p.log_lo;
    // single precision decides away from the bin edges: |ln sigma| of a positive
    // float is below 104, logf is off by less than 1e-6 of it and so are the
    // subtraction and the product, so t32 is within `off` of the position in
    // double precision (whose logarithm is for the few blobs next to an edge)
    if (p.P >= 2 && span > 0.0 && b.sigma > 0.0f && b.sigma < INFINITY) {
        const float inv = (float)((double)p.nbins / span), lo = (float)p.log_lo;
        const float t32 = (logf(b.sigma) - lo) * inv, off = 1e-5f * (104.0f + fabsf(lo)) * inv;
        const float fl = floorf(t32);
        if (t32 - fl > off && fl + 1.0f - t32 > off) return (int)fminf(fmaxf(fl, 0.0f), (float)(p.nbins - 1));
    }
    const double t = (p.P >= 2 && span > 0.0) ? (log((double)b.sigma) - p.log_lo) / span : 0.0;
    double fb = floor((double)p.nbins * t);
    fb = fmin(fmax(fb, 0.0), (double)(p.nbins - 1));
    return (int)fb;
}

__device__ __forceinline__ double blob_volume(float sigma) {
    const double r = 1.4142135623730951 * (double)sigma;
    return 4.0 / 3.0 * 3.141592653589793 * r * r * r;
}


constexpr int PRUNE_THREADS = 1024;
constexpr int NBUCKET = 4096;
enum { ST_UND = 0, ST_IN = 1, ST_OUT = 2 };

__device__ __forceinline__ bool higher(const dog_blob& a, const dog_blob& b) {
    if (a.response != b.response) return a.response > b.response;
    if (a.level != b.level) return a.level < b.level;
    if (a.y != b.y) return a.y < b.y;
    return a.x < b.x;
}

__device__ __forceinline__ int plane_of(const dog_blob& b, int P) { return min(max(b.level, 0), P - 1); }

__device__ __forceinline__ unsigned bucket_of(int cx, int cy) {
    return (((unsigned)cx * 73856093u) ^ ((unsigned)cy * 19349663u)) & (NBUCKET - 1);
}

struct PruneSmem {
    alignas(16) int bcount[NBUCKET];
    alignas(16) int boff[NBUCKET + 1];
    int d2[MAX_LEVELS * MAX_LEVELS];
    int wsum[32];
    int changed;
    int scan_carry;
};

// The buckets of the 3x3 cells around (cx, cy).  Two cells may hash to the
// same bucket; every use below is unaffected by visiting a candidate twice
// (an any-of test, a maximum, a search for the next member in priority order).
__device__ __forceinline__ int neighbour_buckets(int cx, int cy, unsigned* bk) {
    int nb = 0;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) bk[nb++] = bucket_of(cx + dx, cy + dy);
    return nb;
}

// Volume histogram of one frame's pruned blobs (out[0 .. out_count[f])),
// written whole by the frame's CTA (no other CTA touches it).
__device__ void frame_hist(const PruneParams& p, PruneSmem& s, const dog_blob* out, int f) {
    const HistParams& hp = p.hist;
    const int tid = threadIdx.x;
    const int nbo = (hp.mode == DOG_HIST_LADDER) ? hp.P : hp.nbins;
    unsigned* hc = reinterpret_cast<unsigned*>(s.bcount);
    double* hv = reinterpret_cast<double*>(s.boff);
    __syncthreads();
    for (int q = tid; q < nbo; q += PRUNE_THREADS) { hc[q] = 0u; hv[q] = 0.0; }
    __syncthreads();
    const int nout = min(p.out_count[f], p.cap_out);
    for (int i = tid; i < nout; i += PRUNE_THREADS) {
        const dog_blob b = out[i];
        const int bin = hist_bin(b, hp, hp.sig_f, hp.level_bin);
        atomicAdd(&hc[bin], 1u);
        if (hp.vol) atomicAdd(&hv[bin], blob_volume(b.sigma));
    }
    __syncthreads();
    for (int q = tid; q < nbo; q += PRUNE_THREADS) {
        hp.hist[(size_t)f * nbo + q] = hc[q];
        if (hp.vol) hp.vol[(size_t)f * nbo + q] = hv[q];
    }
}

// Exclusive scan of the NBUCKET counts in s.bcount into s.boff (s.boff[NBUCKET]
// the total): four buckets per thread.
static_assert(NBUCKET == 4 * PRUNE_THREADS, "four buckets per thread");
__device__ __forceinline__ void scan_buckets(PruneSmem& s) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int4 c = reinterpret_cast<const int4*>(s.bcount)[tid];
    const int v = c.x + c.y + c.z + c.w;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s.wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = s.wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        s.wsum[lane] = t;
    }
    __syncthreads();
    const int e = x - v + (warp > 0 ? s.wsum[warp - 1] : 0);
    reinterpret_cast<int4*>(s.boff)[tid] = make_int4(e, e + c.x, e + c.x + c.y, e + c.x + c.y + c.z);
    if (tid == PRUNE_THREADS - 1) s.boff[NBUCKET] = e + v;
}

// Frames with at most PRUNE_SMEM_CAND candidates take prune_cells; larger ones, and
// those that it gives back, the hashed cells, with as much of their arrays in
// shared memory as its size allows.
constexpr int PRUNE_SMEM_CAND = 4096;
constexpr int EDGE_WARP = 640;   // conflicts one warp may list

// Shared memory of the frames that fit: the candidates in the order of a grid
// of cells, so that a row of three cells is one contiguous range.
struct CellSmem {
    double hv[DOG_MAX_NBINS], sig[MAX_LEVELS];
    float sig_f[MAX_LEVELS];
    int level_bin[MAX_LEVELS];
    int x[PRUNE_SMEM_CAND], y[PRUNE_SMEM_CAND], level[PRUNE_SMEM_CAND];
    float resp[PRUNE_SMEM_CAND];
    int target[PRUNE_SMEM_CAND];
    unsigned hc[DOG_MAX_NBINS];
    unsigned short cell[PRUNE_SMEM_CAND];
    unsigned char state[PRUNE_SMEM_CAND], in[PRUNE_SMEM_CAND], und[PRUNE_SMEM_CAND];
    union {   // the edges are gone when the members come
        unsigned edge[PRUNE_THREADS / 32 * EDGE_WARP];
        unsigned short member[PRUNE_SMEM_CAND];
    };
    int box[4];   // smallest and largest x and y

    __device__ __forceinline__ bool before(int a, int b) const {   // higher(), by place
        if (resp[a] != resp[b]) return resp[a] > resp[b];
        if (level[a] != level[b]) return level[a] < level[b];
        if (y[a] != y[b]) return y[a] < y[b];
        return x[a] < x[b];
    }
};
constexpr int PRUNE_DYN_BYTES = (int)sizeof(CellSmem);
// hashed cells: the most candidates of which themselves and the three arrays,
// themselves, two arrays and one array fit
constexpr int CAND_FIT = PRUNE_DYN_BYTES / (int)sizeof(dog_blob);
constexpr int PAIR_FIT = PRUNE_DYN_BYTES / 8, ONE_FIT = PRUNE_DYN_BYTES / 4;
constexpr int ALL_FIT = PRUNE_DYN_BYTES / ((int)sizeof(dog_blob) + 3 * (int)sizeof(int));
static_assert(ALL_FIT >= PRUNE_SMEM_CAND, "lists that prune_cells gives back");
static_assert(PRUNE_DYN_BYTES + (int)sizeof(PruneSmem) <= 226 * 1024, "shared memory of one CTA");

// The grid over the candidates' box: cells of at least the largest conflict
// distance, at most NBUCKET of them with a margin of one column on either side.
struct CellGrid {
    long long ox, oy, cell;
    int nx, ny, reach;   // reach: no smaller than any conflict distance squared
};
__device__ __forceinline__ CellGrid cell_grid(const PruneParams& p, const CellSmem& r, int n) {
    CellGrid g;
    g.ox = r.box[0];
    g.oy = r.box[2];
    const long long wx = n ? r.box[1] - g.ox : 0, wy = n ? r.box[3] - g.oy : 0;
    g.cell = p.cell;
    while ((wx / g.cell + 3) * (wy / g.cell + 1) > NBUCKET) g.cell *= 2;
    g.nx = (int)(wx / g.cell) + 3;
    g.ny = (int)(wy / g.cell) + 1;
    g.reach = p.cell < 46340 ? p.cell * p.cell : INT_MAX;
    return g;
}

// Members, blobs and histogram of a frame whose states and targets are settled
// (any: this thread found a target).
__device__ __forceinline__ void finish_cells(const PruneParams& p, PruneSmem& s, CellSmem& r, int n, bool any,
                                             dog_blob* out, int f) {
    const int tid = threadIdx.x, lane = tid & 31;
    const HistParams& hp = p.hist;
    const int nbo = hp.hist ? (hp.mode == DOG_HIST_LADDER ? hp.P : hp.nbins) : 0;
    // members of every accepted candidate (the edges are no longer needed)
    const bool groups = __syncthreads_or(any) && p.mode == DOG_PRUNE_COALESCE;
    if (groups) {
        for (int q = tid; q < NBUCKET; q += PRUNE_THREADS) s.bcount[q] = 0;
        __syncthreads();
        for (int i = tid; i < n; i += PRUNE_THREADS)
            if (r.state[i] == ST_OUT) atomicAdd(&s.bcount[r.target[i]], 1);
        __syncthreads();
        scan_buckets(s);
        __syncthreads();
        for (int i = tid; i < n; i += PRUNE_THREADS)
            if (r.state[i] == ST_OUT) {
                const int t = r.target[i];
                r.member[s.boff[t] + atomicSub(&s.bcount[t], 1) - 1] = (unsigned short)i;
            }
    }
    if (tid == 0) s.scan_carry = s.changed = 0;
    __syncthreads();
    // accepted blobs: compaction and bin
    auto emit = [&](int a, int idx, float sigma) {
        dog_blob o;
        o.x = r.x[a];
        o.y = r.y[a];
        o.level = r.level[a];
        o.sigma = sigma;
        o.response = r.resp[a];
        if (idx < p.cap_out) {
            out[idx] = o;
            if (nbo) {
                const int bin = hist_bin(o, hp, r.sig_f, r.level_bin);
                atomicAdd(&r.hc[bin], 1u);
                if (hp.vol) atomicAdd(&r.hv[bin], blob_volume(sigma));
            }
        } else {
            atomicCAS(p.status, 0, (int)DOG_ERR_CAPACITY);
        }
    };
    for (int a0 = tid & ~31; a0 < n; a0 += PRUNE_THREADS) {
        const int a = a0 + lane;
        const bool acc = a < n && r.state[a] == ST_IN;
        const bool alone = acc && !(groups && s.boff[a + 1] > s.boff[a]);
        const unsigned m = __ballot_sync(0xffffffffu, alone), g = __ballot_sync(0xffffffffu, acc && !alone);
        int idx = 0, gi = 0;
        if (lane == 0 && m) idx = atomicAdd(&s.scan_carry, __popc(m));
        if (lane == 0 && g) gi = atomicAdd(&s.changed, __popc(g));
        idx = __shfl_sync(0xffffffffu, idx, 0) + __popc(m & ((1u << lane) - 1u));
        gi = __shfl_sync(0xffffffffu, gi, 0) + __popc(g & ((1u << lane) - 1u));
        if (alone) emit(a, idx, (float)r.sig[min(max(r.level[a], 0), p.P - 1)]);
        else if (acc) r.target[gi] = a;   // (targets are in the member lists now)
    }
    if (groups) {
        // groups: mean sigma summed in visiting order.  Gathered in a list, so that
        // the double-precision instructions (two lanes a cycle and SM) run in few
        // full warps and not in every warp that has a group
        __syncthreads();
        const int ng = s.changed, first = s.scan_carry;
        for (int q = tid; q < ng; q += PRUNE_THREADS) {
            const int a = r.target[q];
            const int m0 = s.boff[a], m1 = s.boff[a + 1];
            for (int u = m0 + 1; u < m1; ++u) {   // by priority (few members)
                const unsigned short v = r.member[u];
                int w = u;
                for (; w > m0 && r.before(v, r.member[w - 1]); --w) r.member[w] = r.member[w - 1];
                r.member[w] = v;
            }
            const int la = min(max(r.level[a], 0), p.P - 1);
            double sum = r.sig[la];
            bool mixed = false;
            for (int u = m0; u < m1; ++u) {
                const int lv = r.level[r.member[u]];
                sum += r.sig[min(max(lv, 0), p.P - 1)];
                mixed |= lv != r.level[a];
            }
            emit(a, first + q, mixed ? (float)(sum / (double)(1 + m1 - m0)) : (float)r.sig[la]);
        }
        __syncthreads();
        if (tid == 0) s.scan_carry += ng;
    }
    __syncthreads();
    if (tid == 0) p.out_count[f] = s.scan_carry;
    for (int q = tid; q < nbo; q += PRUNE_THREADS) {
        hp.hist[(size_t)f * nbo + q] = r.hc[q];
        if (hp.vol) hp.vol[(size_t)f * nbo + q] = r.hv[q];
    }
}

// Pruning and histogram of one frame in shared memory.  One thread per
// candidate walking its nine hashed cells, once a round and once per group
// member, is a chain of dependent loads as long as the fullest cell among 32
// lanes, and the histogram's passes over global memory come on top (69 us for
// the 1,700 candidates of a 1024 x 1024 frame).  Here the candidates are copied
// in the order of a plain grid, the conflicts (few: 2 to 5% of the candidates on
// PLIF frames) are listed once as edges (candidate, higher-priority neighbour),
// the rounds, targets and members run over the edges, and the accepted blobs are
// binned as they are written.  (Sorting by priority instead, so that it becomes
// an integer comparison, took 17 us for the sort alone.)  Returns CELLS_FULL when a
// warp finds more than EDGE_WARP conflicts (the candidates are sorted: dense_cells
// goes on from there), and CELLS_FAR, having written nothing, when the candidates
// lie too far apart for the grid.
enum { CELLS_DONE = 0, CELLS_FULL = 1, CELLS_FAR = 2 };
__device__ __forceinline__ int prune_cells(const PruneParams& p, PruneSmem& s, CellSmem& r, const dog_blob* cand,
                                            int n, dog_blob* out, int f) {
    const int tid = threadIdx.x, lane = tid & 31;
    const HistParams& hp = p.hist;
    const int nbo = hp.hist ? (hp.mode == DOG_HIST_LADDER ? hp.P : hp.nbins) : 0;
    for (int q = tid; q < NBUCKET; q += PRUNE_THREADS) s.bcount[q] = 0;
    for (int q = tid; q < p.P * p.P; q += PRUNE_THREADS) s.d2[q] = p.d2thr[q];
    for (int q = tid; q < p.P; q += PRUNE_THREADS) {
        r.sig[q] = p.sig[q];
        r.sig_f[q] = hp.hist ? hp.sig_f[q] : 0.0f;
        r.level_bin[q] = hp.hist ? hp.level_bin[q] : 0;
    }
    for (int q = tid; q < nbo; q += PRUNE_THREADS) { r.hc[q] = 0u; r.hv[q] = 0.0; }
    if (tid < 4) r.box[tid] = tid & 1 ? INT_MIN : INT_MAX;
    // this thread's candidates: tid, tid + 1024, ...
    constexpr int PER = PRUNE_SMEM_CAND / PRUNE_THREADS;
    dog_blob mine[PER];
    int bk[PER];
    int x0 = INT_MAX, x1 = INT_MIN, y0 = INT_MAX, y1 = INT_MIN;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int i = tid + u * PRUNE_THREADS;
        if (i < n) {
            mine[u] = cand[i];
            x0 = min(x0, mine[u].x); x1 = max(x1, mine[u].x);
            y0 = min(y0, mine[u].y); y1 = max(y1, mine[u].y);
        }
    }
    x0 = __reduce_min_sync(0xffffffffu, x0); x1 = __reduce_max_sync(0xffffffffu, x1);
    y0 = __reduce_min_sync(0xffffffffu, y0); y1 = __reduce_max_sync(0xffffffffu, y1);
    __syncthreads();
    if (lane == 0) {
        atomicMin(&r.box[0], x0); atomicMax(&r.box[1], x1);
        atomicMin(&r.box[2], y0); atomicMax(&r.box[3], y1);
    }
    __syncthreads();
    const CellGrid g = cell_grid(p, r, n);
    const long long ox = g.ox, oy = g.oy, cell = g.cell;
    const int nx = g.nx, ny = g.ny;
    // (candidates of neighbouring cells are less than two cells apart; of cells
    // this large, in frames of more than 2^24 rows, the squared distance would not
    // fit an int)
    if (cell > 16384) return CELLS_FAR;
    const unsigned uc = (unsigned)cell;   // (at most the extent, below 2^32)
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (tid + u * PRUNE_THREADS < n) {
            bk[u] = (int)((unsigned)(mine[u].y - oy) / uc) * nx + (int)((unsigned)(mine[u].x - ox) / uc) + 1;
            atomicAdd(&s.bcount[bk[u]], 1);
        }
    __syncthreads();
    scan_buckets(s);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (tid + u * PRUNE_THREADS < n) {
            const int at = s.boff[bk[u]] + atomicSub(&s.bcount[bk[u]], 1) - 1;
            r.x[at] = mine[u].x;
            r.y[at] = mine[u].y;
            r.level[at] = mine[u].level;
            r.resp[at] = mine[u].response;
            r.cell[at] = (unsigned short)bk[u];
            r.target[at] = -1;
            r.state[at] = ST_UND;
            r.in[at] = 0;
            r.und[at] = 0;
        }
    __syncthreads();
    // edges: candidate i and row of cells dy - 1 per thread; every warp fills and
    // later reads its own part of the list (hits are rare, so they may diverge)
    unsigned* edge = r.edge + (tid >> 5) * EDGE_WARP;
    int* n_edge = &s.wsum[tid >> 5];
    if (lane == 0) *n_edge = 0;
    __syncwarp();
    const int reach = g.reach;
    for (int t = tid; t < 3 * n; t += PRUNE_THREADS) {
        const int dy = (t >= n) + (t >= 2 * n), i = t - dy * n;
        const int xi = r.x[i], yi = r.y[i];
        const int c = r.cell[i] + (dy - 1) * nx;
        if (c < 0 || c >= nx * ny) continue;
        const int end = s.boff[c + 2];
        for (int k = s.boff[c - 1]; k < end; ++k) {
            const int ex = r.x[k] - xi, ey = r.y[k] - yi, d = ex * ex + ey * ey;
            if (d >= reach || k == i) continue;
            const int li = min(max(r.level[i], 0), p.P - 1), lk = min(max(r.level[k], 0), p.P - 1);
            if (d >= s.d2[li * p.P + lk] || !r.before(k, i)) continue;
            const int e = atomicAdd(n_edge, 1);
            if (e < EDGE_WARP) edge[e] = (unsigned)i << 16 | (unsigned)k;
        }
    }
    __syncwarp();
    const int ne = *n_edge;
    if (__syncthreads_or(ne > EDGE_WARP)) return CELLS_FULL;
    // rounds of the independent-set rule
    for (;;) {
        for (int e = lane; e < ne; e += 32) {
            const int i = edge[e] >> 16;
            if (r.state[i] != ST_UND) continue;
            const int st = r.state[edge[e] & 0xffffu];
            if (st == ST_IN) r.in[i] = 1;
            else if (st == ST_UND) r.und[i] = 1;
        }
        __syncthreads();
        bool wait = false;
        for (int i = tid; i < n; i += PRUNE_THREADS) {
            if (r.state[i] != ST_UND) continue;
            if (r.in[i] || !r.und[i]) r.state[i] = r.in[i] ? ST_OUT : ST_IN;
            else wait = true;
            r.und[i] = 0;
        }
        if (!__syncthreads_or(wait)) break;   // (each round settles the first undecided)
    }
    // every rejected candidate joins its highest-priority accepted neighbour
    bool any = false;
    for (int e = lane; e < ne; e += 32) {
        const int i = edge[e] >> 16, j = edge[e] & 0xffffu;
        if (r.state[i] != ST_OUT || r.state[j] != ST_IN) continue;
        any = true;
        int seen = r.target[i];
        while (seen < 0 || r.before(j, seen)) {
            const int now = atomicCAS(&r.target[i], seen, j);
            if (now == seen) break;
            seen = now;
        }
    }
    finish_cells(p, s, r, n, any, out, f);
    return CELLS_DONE;
}

// The frame of prune_cells' CELLS_FULL: every round, and then the targets, walk the
// rows of cells again.  A state is settled once, so a round may see others before
// or after theirs.  Out of line and apart, so that the frames without need are not
// compiled for it (with both in prune_cells a frame of the FFT backend took 29.3 us
// in place of 20.6; apart 21.3).
__device__ __noinline__ void dense_cells(const PruneParams& p, PruneSmem& s, CellSmem& r, int n, dog_blob* out, int f) {
    const CellGrid g = cell_grid(p, r, n);
    const int nx = g.nx, ny = g.ny, reach = g.reach;
    auto walk = [&](int i, auto visit) {   // i's neighbours of higher priority, until visit() has seen enough
        const int xi = r.x[i], yi = r.y[i], li = min(max(r.level[i], 0), p.P - 1);
        for (int dy = -1; dy <= 1; ++dy) {
            const int c = r.cell[i] + dy * nx;
            if (c < 0 || c >= nx * ny) continue;
            const int end = s.boff[c + 2];
            for (int k = s.boff[c - 1]; k < end; ++k) {
                const int ex = r.x[k] - xi, ey = r.y[k] - yi, d = ex * ex + ey * ey;
                if (d >= reach || k == i) continue;
                if (d < s.d2[li * p.P + min(max(r.level[k], 0), p.P - 1)] && r.before(k, i) && visit(k)) return;
            }
        }
    };
    volatile unsigned char* state = r.state;
    for (;;) {
        bool wait = false;
        for (int i = threadIdx.x; i < n; i += PRUNE_THREADS) {
            if (state[i] != ST_UND) continue;
            bool in = false, und = false;
            walk(i, [&](int k) {
                const int st = state[k];
                und |= st == ST_UND;
                return in = st == ST_IN;
            });
            if (in || !und) state[i] = in ? ST_OUT : ST_IN;
            else wait = true;
        }
        if (!__syncthreads_or(wait)) break;
    }
    bool any = false;
    for (int i = threadIdx.x; i < n; i += PRUNE_THREADS) {
        if (r.state[i] != ST_OUT) continue;
        int best = -1;
        walk(i, [&](int k) {
            if (r.state[k] == ST_IN && (best < 0 || r.before(k, best))) best = k;
            return false;
        });
        r.target[i] = best;
        any = true;
    }
    finish_cells(p, s, r, n, any, out, f);
}

__global__ void __launch_bounds__(PRUNE_THREADS) dog_prune_kernel(const __grid_constant__ PruneParams p) {
    __shared__ PruneSmem s;
    extern __shared__ int4 prune_dyn[];
    const int f = blockIdx.x;
    const int tid = threadIdx.x;
    const long long coff = p.cand_off ? p.cand_off[f] : 0;
    const long long ooff = p.out_off ? p.out_off[f] : 0;
    const dog_blob* cand = p.cand + coff;
    int* state = p.state + coff;
    int* target = p.target + coff;
    int* order = p.order + coff;
    dog_blob* out = p.out + ooff;
    const int n = min(p.cand_count[f], p.cap_in);
    if (p.mode != DOG_PRUNE_OFF) {
        if (n <= PRUNE_SMEM_CAND) {
            CellSmem& r = *reinterpret_cast<CellSmem*>(prune_dyn);
            const int got = prune_cells(p, s, r, cand, n, out, f);
            if (got == CELLS_FULL) dense_cells(p, s, r, n, out, f);
            if (got != CELLS_FAR) return;
            __syncthreads();
        }
        // Copies in the shared memory that the launch has anyway, and that leaves the
        // L1 too small for these arrays in global memory (5000 candidates 820 us, with
        // 60 KB less of it 706, copied 381): the candidates and all three arrays up to
        // 5872 of them, the candidates up to 9396; of longer lists the arrays that the
        // inner loops read most, up to 23490 and 46980 (23,000: 8095, 7740, 5611).
        int* si = reinterpret_cast<int*>(prune_dyn);
        if (n <= CAND_FIT) {
            dog_blob* sc = reinterpret_cast<dog_blob*>(prune_dyn);
            for (int i = tid; i < n; i += PRUNE_THREADS) sc[i] = cand[i];
            cand = sc;
            si = reinterpret_cast<int*>(sc + n);
        }
        if (n <= ALL_FIT) {
            state = si;
            target = si + n;
            order = si + 2 * n;
        } else if (n > CAND_FIT && n <= PAIR_FIT) {
            state = si;
            order = si + n;
        } else if (n > CAND_FIT && n <= ONE_FIT) {
            state = si;
        }
        // made visible by the first __syncthreads below
    }

    if (p.mode == DOG_PRUNE_OFF) {
        for (int i = tid; i < n; i += PRUNE_THREADS) {
            if (i < p.cap_out) out[i] = cand[i];
        }
        if (tid == 0) {
            p.out_count[f] = n;
            if (n > p.cap_out) atomicCAS(p.status, 0, (int)DOG_ERR_CAPACITY);
        }
        if (p.hist.hist) frame_hist(p, s, out, f);
        return;
    }

    for (int q = tid; q < NBUCKET; q += PRUNE_THREADS) s.bcount[q] = 0;
    for (int q = tid; q < p.P * p.P; q += PRUNE_THREADS) s.d2[q] = p.d2thr[q];
    if (tid == 0) p.out_count[f] = 0;
    __syncthreads();
    const int cell = p.cell;

    // 1. counting sort of candidate indices by hashed cell
    for (int i = tid; i < n; i += PRUNE_THREADS) {
        const dog_blob b = cand[i];
        const unsigned bk = bucket_of(b.x / cell, b.y / cell);
        target[i] = (int)bk;
        atomicAdd(&s.bcount[bk], 1);
        state[i] = ST_UND;
    }
    __syncthreads();
    scan_buckets(s);
    __syncthreads();
    for (int q = tid; q < NBUCKET; q += PRUNE_THREADS) s.bcount[q] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += PRUNE_THREADS) {
        const int bk = target[i];
        const int pos = s.boff[bk] + atomicAdd(&s.bcount[bk], 1);
        order[pos] = i;
    }
    __syncthreads();

    // 2. rounds of the independent-set rule
    volatile int* vstate = state;
    for (int round = 0; round <= n + 1; ++round) {
        if (tid == 0) s.changed = 0;
        __syncthreads();
        for (int i = tid; i < n; i += PRUNE_THREADS) {
            if (vstate[i] != ST_UND) continue;
            const dog_blob bi = cand[i];
            unsigned bk[9];
            neighbour_buckets(bi.x / cell, bi.y / cell, bk);
            bool any_in = false, any_und = false;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                if (any_in) break;
                for (int k = s.boff[bk[q]]; k < s.boff[bk[q] + 1]; ++k) {
                    const int j = order[k];
                    if (j == i) continue;
                    const dog_blob bj = cand[j];
                    const int dx = bj.x - bi.x, dy = bj.y - bi.y;
                    if (dx * dx + dy * dy >= s.d2[plane_of(bi, p.P) * p.P + plane_of(bj, p.P)]) continue;
                    if (!higher(bj, bi)) continue;
                    const int st = vstate[j];
                    if (st == ST_IN) { any_in = true; break; }
                    if (st == ST_UND) any_und = true;
                }
            }
            if (any_in) { vstate[i] = ST_OUT; s.changed = 1; }
            else if (!any_und) { vstate[i] = ST_IN; s.changed = 1; }
        }
        __syncthreads();
        if (!s.changed) break;
        __syncthreads();
    }

    // 3. every rejected candidate joins its highest-priority accepted neighbour
    for (int i = tid; i < n; i += PRUNE_THREADS) {
        target[i] = -1;
        if (state[i] != ST_OUT) continue;
        const dog_blob bi = cand[i];
        unsigned bk[9];
        neighbour_buckets(bi.x / cell, bi.y / cell, bk);
        int best = -1;
#pragma unroll
        for (int q = 0; q < 9; ++q)
            for (int k = s.boff[bk[q]]; k < s.boff[bk[q] + 1]; ++k) {
                const int j = order[k];
                if (j == i || (state[j] & 3) != ST_IN) continue;
                const dog_blob bj = cand[j];
                const int dx = bj.x - bi.x, dy = bj.y - bi.y;
                if (dx * dx + dy * dy >= s.d2[plane_of(bi, p.P) * p.P + plane_of(bj, p.P)]) continue;
                if (!higher(bj, bi)) continue;
                if (best < 0 || higher(bj, cand[best])) best = j;
            }
        target[i] = best;
        if (best < 0) atomicCAS(p.status, 0, (int)DOG_ERR_INVALID);   // cannot happen
        else atomicAdd(&state[best], 4);   // member count of an accepted candidate, above the state bits
    }
    __syncthreads();

    // 4. accepted blobs: group mean sigma summed in visiting order, then compaction
    for (int a = tid; a < n; a += PRUNE_THREADS) {
        if ((state[a] & 3) != ST_IN) continue;
        const int nmem = state[a] >> 2;
        const dog_blob ba = cand[a];
        double sum = p.sig[plane_of(ba, p.P)];
        int cnt = 1;
        bool mixed = false;
        if (p.mode == DOG_PRUNE_COALESCE && nmem > 0) {
            unsigned bk[9];
            neighbour_buckets(ba.x / cell, ba.y / cell, bk);
            int prev = a;
            for (;;) {
                // next member after `prev` in priority order
                int nxt = -1;
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    for (int k = s.boff[bk[q]]; k < s.boff[bk[q] + 1]; ++k) {
                        const int j = order[k];
                        if (target[j] != a) continue;
                        const dog_blob bj = cand[j];
                        if (!higher(cand[prev], bj)) continue;
                        if (nxt < 0 || higher(bj, cand[nxt])) nxt = j;
                    }
                if (nxt < 0) break;
                const dog_blob bn = cand[nxt];
                sum += p.sig[plane_of(bn, p.P)];
                ++cnt;
                mixed |= (bn.level != ba.level);
                prev = nxt;
                if (cnt > nmem) break;   // all members visited
            }
        }
        dog_blob o = ba;
        o.sigma = mixed ? (float)(sum / (double)cnt) : (float)p.sig[plane_of(ba, p.P)];
        const int idx = atomicAdd(&p.out_count[f], 1);
        if (idx < p.cap_out) out[idx] = o;
        else atomicCAS(p.status, 0, (int)DOG_ERR_CAPACITY);
    }
    // 5. optional: this frame's volume histogram
    if (p.hist.hist) frame_hist(p, s, out, f);
}

// Set once per device (not on every launch, so launches can be graph-captured);
// atomic because the launcher may be called from several host threads.
static std::atomic<bool> g_prune_attr[64];

cudaError_t launch_prune(const PruneParams& p, cudaStream_t s) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!g_prune_attr[dev & 63].load(std::memory_order_acquire)) {
        // setting the attribute twice from two threads is harmless
        e = cudaFuncSetAttribute(dog_prune_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PRUNE_DYN_BYTES);
        if (e != cudaSuccess) return e;
        g_prune_attr[dev & 63].store(true, std::memory_order_release);
    }
    dog_prune_kernel<<<p.n_frames, PRUNE_THREADS, PRUNE_DYN_BYTES, s>>>(p);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Histogram: one CTA row per frame, shared-memory bins, one global atomic per
// non-empty bin and CTA.
__global__ void __launch_bounds__(256) dog_hist_kernel(const __grid_constant__ HistParams p) {
    __shared__ unsigned hc[DOG_MAX_NBINS];
    __shared__ double hv[DOG_MAX_NBINS];
    const int f = blockIdx.y;
    const int nbo = (p.mode == DOG_HIST_LADDER) ? p.P : p.nbins;
    for (int q = threadIdx.x; q < nbo; q += blockDim.x) { hc[q] = 0u; hv[q] = 0.0; }
    __syncthreads();
    const long long off = p.off ? p.off[f] : 0;
    const int n = min(p.count[f], p.cap);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const dog_blob b = p.blobs[off + i];
        const int bin = hist_bin(b, p, p.sig_f, p.level_bin);
        atomicAdd(&hc[bin], 1u);
        if (p.vol) atomicAdd(&hv[bin], blob_volume(b.sigma));
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nbo; q += blockDim.x) {
        if (hc[q]) atomicAdd(&p.hist[(size_t)f * nbo + q], hc[q]);
        if (p.vol && hv[q] != 0.0) atomicAdd(&p.vol[(size_t)f * nbo + q], hv[q]);
    }
}

cudaError_t launch_hist(const HistParams& p, cudaStream_t s) {
    dim3 grid(4, p.n_frames);
    dog_hist_kernel<<<grid, 256, 0, s>>>(p);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
__global__ void dog_ring_push_kernel(const uint32_t* hist, int nbins, uint32_t* ring, int window,
                                     uint32_t* sum, int32_t* head) {
    const int h = *head;
    const int slot = ((h % window) + window) % window;
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        const uint32_t old = (h >= window) ? ring[(size_t)slot * nbins + b] : 0u;
        const uint32_t nw = hist[b];
        ring[(size_t)slot * nbins + b] = nw;
        sum[b] = sum[b] - old + nw;
    }
    __syncthreads();
    if (threadIdx.x == 0) *head = h + 1;
}

cudaError_t launch_ring_push(const uint32_t* hist, int nbins, uint32_t* ring, int window, uint32_t* sum,
                             int32_t* head, cudaStream_t s) {
    dog_ring_push_kernel<<<1, 256, 0, s>>>(hist, nbins, ring, window, sum, head);
    return cudaGetLastError();
}

// One CTA per stream walks the batch in order and pushes that stream's frames.
__global__ void dog_ring_push_batched_kernel(const uint32_t* hists, const int32_t* ids, int n, int nbins,
                                             uint32_t* rings, int window, uint32_t* sums, int32_t* heads) {
    const int sid = blockIdx.x;
    uint32_t* ring = rings + (size_t)sid * window * nbins;
    uint32_t* sum = sums + (size_t)sid * nbins;
    int h = heads[sid];
    for (int f = 0; f < n; ++f) {
        if (ids[f] != sid) continue;
        const int slot = h % window;
        for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
            const uint32_t old = (h >= window) ? ring[(size_t)slot * nbins + b] : 0u;
            const uint32_t nw = hists[(size_t)f * nbins + b];
            ring[(size_t)slot * nbins + b] = nw;
            sum[b] = sum[b] - old + nw;
        }
        ++h;
        __syncthreads();
    }
    if (threadIdx.x == 0) heads[sid] = h;
}

cudaError_t launch_ring_push_batched(const uint32_t* hists, const int32_t* ids, int n, int nbins, int n_streams,
                                     uint32_t* rings, int window, uint32_t* sums, int32_t* heads, cudaStream_t s) {
    dog_ring_push_batched_kernel<<<n_streams, 128, 0, s>>>(hists, ids, n, nbins, rings, window, sums, heads);
    return cudaGetLastError();
}

}  // namespace dogk

// build.cu -- octree construction on the GPU: bounding cube, Morton keys,
// stable LSD radix sort, gather into key order, topology, walk groups and
// cell multipoles (monopole + traceless quadrupole about the centre of mass,
// the expansion a tree code uses for distant groups, Sect. 1).
//
// Topology without per-level launches: for sorted keys, let D(j) be the first
// level at which key[j-1] and key[j] differ (D(0) = D(n) = 0, 22 for equal
// keys). At level l the key prefixes cut the sorted array at the positions
// with D(j) <= l. A star i lies in a cell at level l iff every coarser cell
// holding it has more than n_leaf stars, i.e. iff l <= lambda_i, the first
// level whose segment around i holds at most n_leaf stars (capped at 21).
// lambda_i only depends on D within n_leaf positions of i, so one pass over
// a window finds it; cells starting at i are levels D(i)..lambda_i, and their
// breadth-first index (level, first star) comes from per-level ballots and
// one flat scan.
#include <algorithm>

#include "rv_internal.cuh"

namespace rv {

// ---------------------------------------------------------------------------
// block helpers
// ---------------------------------------------------------------------------
template <int NT>
__device__ __forceinline__ int block_exclusive_scan(int v, int *smem_warp, int &total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) smem_warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int w = (lane < NT / 32) ? smem_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < NT / 32) smem_warp[lane] = w;
    }
    __syncthreads();
    int warp_base = (wid > 0) ? smem_warp[wid - 1] : 0;
    total = smem_warp[NT / 32 - 1];
    __syncthreads();
    return warp_base + x - v;
}

// ---------------------------------------------------------------------------
// Single-pass scans over tiles ("decoupled look-back": Merrill & Garland 2016).
// A block takes the next tile from a ticket counter, publishes its tile's sum,
// adds up its predecessors' published words back to the nearest full prefix,
// and publishes its own prefix. A tile's predecessors have always started (the
// tickets are handed out in order), so every wait ends; waits are bounded all
// the same, and a block that gives up latches RV_E_TIMEOUT and writes nothing;
// what it leaves unwritten is not used: a sort sets the kLbGaveUp word, which the
// kernels after it read, a scan or the group pass leaves a total of -1.
// A word holds its state in the top two bits (0: not there yet) and the count
// below (counts stay under 2^30), so that one store publishes both.
// ---------------------------------------------------------------------------
constexpr unsigned kLbSum = 1u << 30, kLbPrefix = 2u << 30, kLbCount = (1u << 30) - 1;
constexpr int kLbSpins = 1 << 20;   // polls before a wait gives up (about half a second)

__device__ __forceinline__ unsigned lb_load(const unsigned *p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void lb_store(unsigned *p, unsigned v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The sum of the tiles before `tile` (one word a tile), by one whole warp: 32
// predecessors a step. Returns false if a wait gave up.
__device__ __forceinline__ bool lb_sum_before(const unsigned *words, int tile, int polls, unsigned &sum) {
    const int lane = threadIdx.x & 31;
    sum = 0;
    for (int hi = tile - 1; hi >= 0; hi -= 32) {
        const int t = hi - lane;
        unsigned w = t >= 0 ? lb_load(words + t) : kLbPrefix;   // before the first tile: a prefix of 0
        for (int spin = 0; __any_sync(0xffffffffu, (w >> 30) == 0); spin++) {
            if (spin > polls) return false;
            if ((w >> 30) == 0) w = lb_load(words + t);
        }
        const unsigned pm = __ballot_sync(0xffffffffu, w & kLbPrefix);
        const int stop = pm ? __ffs(pm) - 1 : 31;   // the nearest prefix ends the search
        sum += __reduce_add_sync(0xffffffffu, lane <= stop ? w & kLbCount : 0u);
        if (pm) break;
    }
    return true;
}

// The total of a pass by look-back, 0 before the launch: the last tile's sum, or
// -1 once any tile gave up, in whichever order they end.
__device__ __forceinline__ void lb_total(int *d_total, bool ok, bool last, int total) {
    if (!ok) atomicExch(d_total, -1);
    else if (last) atomicCAS(d_total, 0, total);
}

// Exclusive scan of n int32 in place; the total to *d_total (lb_total). words, ticket: zero before the launch. gave_up
// (optional): set if the data is not there, and then nothing is done.
__global__ void __launch_bounds__(256) scan_k(int *data, int64_t len, unsigned *words, int *ticket,
                                              const unsigned *gave_up, LbWait wait, int *d_total, DevState *st) {
    __shared__ int sw[8], stile;
    __shared__ unsigned sbefore;
    __shared__ bool sok;
    if (threadIdx.x == 0) {
        const int t = atomicAdd(ticket, 1);
        stile = gave_up && lb_load(gave_up) ? -1 : t;
    }
    __syncthreads();
    const int tile = stile;
    if (tile < 0) return;
    const int64_t base = (int64_t)tile * kScanChunk + threadIdx.x * 8;
    int v[8], s = 0;
    if (base + 8 <= len) {   // the tile's start is 32-byte aligned
        const int4 a = *reinterpret_cast<const int4 *>(data + base), b = *reinterpret_cast<const int4 *>(data + base + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = (base + k < len) ? data[base + k] : 0;
    }
#pragma unroll
    for (int k = 0; k < 8; k++) s += v[k];
    int total;
    const int ex0 = block_exclusive_scan<256>(s, sw, total);
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0 && tile != wait.hold)
            lb_store(words + tile, (tile ? kLbSum : kLbPrefix) | (unsigned)total);
        unsigned before = 0;
        const bool ok = lb_sum_before(words, tile, wait.polls, before);
        if (threadIdx.x == 0) {
            if (ok && tile) lb_store(words + tile, kLbPrefix | ((before + (unsigned)total) & kLbCount));
            if (!ok) latch_err(st, kErrLookback);
            sbefore = before;
            sok = ok;
            lb_total(d_total, ok, tile == (int)gridDim.x - 1, (int)before + total);
        }
    }
    __syncthreads();
    if (!sok) return;
    int ex = ex0 + (int)sbefore;
    int o[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
        o[k] = ex;
        ex += v[k];
    }
    if (base + 8 <= len) {
        *reinterpret_cast<int4 *>(data + base) = make_int4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<int4 *>(data + base + 4) = make_int4(o[4], o[5], o[6], o[7]);
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++)
            if (base + k < len) data[base + k] = o[k];
    }
}

// The wait of a stage's next launch (the self-test's, once, if it named this stage).
static LbWait lb_wait(rv_ctx *c, int stage) {
    if (c->lb_test_stage != stage) return LbWait{kLbSpins, -1};
    c->lb_test_stage = 0;
    return LbWait{c->lb_test_polls, 0};
}

static rv_status scan_launch(rv_ctx *c, int *data, int64_t n, int *d_total, unsigned *words, int *ticket,
                             const unsigned *gave_up, cudaStream_t s) {
    scan_k<<<ceil_div(n, kScanChunk), 256, 0, s>>>(data, n, words, ticket, gave_up, lb_wait(c, kLbStageScan), d_total,
                                                   c->w.st);
    count_launch(c);
    return cuda_check(c, cudaGetLastError(), "scan");
}

// *d_total is 0 before; -1 after it means that a wait gave up.
rv_status exclusive_scan(rv_ctx *c, int *data, int64_t n, int *d_total, cudaStream_t s) {
    if (n <= 0) return RV_OK;
    // ticket and words side by side: one clear
    unsigned *z = c->w.lb + kLbScan;
    rv_status r = cuda_check(c, cudaMemsetAsync(z, 0, sizeof(unsigned) * (1 + (size_t)ceil_div(n, kScanChunk)), s),
                             "scan");
    if (r != RV_OK) return r;
    return scan_launch(c, data, n, d_total, z + 1, reinterpret_cast<int *>(z), nullptr, s);
}

// ---------------------------------------------------------------------------
// bounding cube
// ---------------------------------------------------------------------------
// The bounding cube of an axis-wise range: min x, y, z; L = max_a (max_a - min_a)
// with FP64 differences; scale = 2^21 / L (0 if L = 0).
__device__ __forceinline__ void cube_of(const float lo[3], const float hi[3], double out[5]) {
    double L = 0.0;
    for (int a = 0; a < 3; a++) {
        bool empty = !(lo[a] <= hi[a]);
        double e = empty ? 0.0 : __dsub_rn((double)hi[a], (double)lo[a]);
        if (e > L) L = e;
        out[a] = empty ? 0.0 : (double)lo[a];
    }
    out[3] = L;
    out[4] = (L > 0.0) ? __ddiv_rn(2097152.0, L) : 0.0;
}

// Blocks (bx, m): member m's stars, strided by bpm blocks; the last block of a
// member to finish reduces the blocks' partials (min and max are exact, so the
// order is free). The first kernel of a build, it also clears the words the
// later ones count in (zero[nzero]), the member roots and the last build's sizes.
//
// n and the members' number are the launch's own, the offsets are read from the
// workspace: a caller's graph that is replayed after another build finds that
// build's offsets there. Then the digit counts would not be those of the n keys
// that are sorted, so the build is given up (offsets_fit) and no star is read
// beyond n.
__device__ __forceinline__ bool offsets_fit(const int64_t *moff, int M, int64_t n) {   // by one block
    bool bad = threadIdx.x == 0 && (moff[0] != 0 || moff[M] != n);
    for (int k = threadIdx.x; k < M; k += blockDim.x) bad |= moff[k] > moff[k + 1];
    return !__syncthreads_or(bad);
}

__global__ void __launch_bounds__(256) bounds_k(int64_t n, const int64_t *moff, int bpm, const float *x, const float *y,
                                                const float *z, float *part, int *arrive, double *mbounds,
                                                DevState *st, unsigned *zero, int64_t nzero, int *mroot) {
    const int m = blockIdx.y;
    const int64_t nthr = (int64_t)gridDim.x * gridDim.y * 256;
    const int64_t tid = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 256 + threadIdx.x;
    for (int64_t i = tid; i < nzero; i += nthr) zero[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        mroot[m] = -1;
        if (m == 0) st->ncell = st->ngroup = 0;
    }
    if (blockIdx.x == 0 && m == 0 && !offsets_fit(moff, gridDim.y, n) && threadIdx.x == 0) {
        latch_err(st, kErrOffsets);
        zero[kLbGaveUp] = 1;   // (after this block's clear of it, above)
    }
    const int64_t s = max(moff[m], (int64_t)0), e = min(moff[m + 1], n);
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = s + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < e; i += (int64_t)bpm * blockDim.x) {
        float v[3] = {x[i], y[i], z[i]};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            lo[a] = fminf(lo[a], v[a]);
            hi[a] = fmaxf(hi[a], v[a]);
        }
    }
    __shared__ float sh[8][6];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto warp_minmax = [&]() {
#pragma unroll
        for (int a = 0; a < 3; a++)
            for (int o = 16; o > 0; o >>= 1) {
                lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
                hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
            }
    };
    warp_minmax();
    if (lane == 0)
        for (int a = 0; a < 3; a++) { sh[wid][a] = lo[a]; sh[wid][3 + a] = hi[a]; }
    __syncthreads();
    if (threadIdx.x < 6) {
        float r = sh[0][threadIdx.x];
        for (int w = 1; w < 8; w++)
            r = (threadIdx.x < 3) ? fminf(r, sh[w][threadIdx.x]) : fmaxf(r, sh[w][threadIdx.x]);
        part[6 * ((int64_t)m * bpm + blockIdx.x) + threadIdx.x] = r;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(arrive + m, 1) == bpm - 1;
        if (last) arrive[m] = 0;   // ready for the next build
        __threadfence();
    }
    __syncthreads();
    if (!last || wid != 0) return;
    for (int a = 0; a < 3; a++) { lo[a] = INFINITY; hi[a] = -INFINITY; }
    for (int b = lane; b < bpm; b += 32)
        for (int a = 0; a < 3; a++) {
            lo[a] = fminf(lo[a], __ldcg(&part[6 * ((int64_t)m * bpm + b) + a]));
            hi[a] = fmaxf(hi[a], __ldcg(&part[6 * ((int64_t)m * bpm + b) + 3 + a]));
        }
    warp_minmax();
    if (lane != 0) return;
    double out[5];
    cube_of(lo, hi, out);
    for (int k = 0; k < 5; k++) {
        mbounds[5 * m + k] = out[k];
        if (m == 0) st->bounds[k] = out[k];
    }
}

// ---------------------------------------------------------------------------
// Morton keys
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x1f00000000ffffull;
    x = (x | (x << 16)) & 0x1f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

__device__ __forceinline__ uint32_t compact3(uint64_t x) {
    x &= 0x1249249249249249ull;
    x = (x | (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x | (x >> 4)) & 0x100f00f00f00f00full;
    x = (x | (x >> 8)) & 0x1f0000ff0000ffull;
    x = (x | (x >> 16)) & 0x1f00000000ffffull;
    x = (x | (x >> 32)) & 0x1fffffull;
    return (uint32_t)x;
}

// q = min(floor((x - min) * scale), 2^21 - 1): one FP64 subtraction, one FP64
// product; for 0 <= t < 2^21 - 1 the floor is the conversion toward zero.
__device__ __forceinline__ uint32_t grid_coord(float v, double lo, double scale) {
    const double t = __dmul_rn(__dsub_rn((double)v, lo), scale);
    if (!(t >= 0.0)) return 0u;
    if (t >= 2097151.0) return 2097151u;
    return (uint32_t)__double2uint_rz(t);
}

// The same q decided in FP32 where FP32 can decide it (GB300's FP64 rate is
// a small fraction of its FP32 rate, and the FP64 rule bound the key kernel).
// d = x - min is formed exactly as an unevaluated pair of floats dh + dl
// (Knuth's two-sum), scale as the pair sh + sl (sl the FP32 rounding of the
// FP64 difference scale - sh, itself exact), and d * scale as ph + c: ph =
// dh sh rounded, its rounding error recovered exactly by an FMA, the cross
// terms dh sl and dl sh added by FMAs, dl sl left out. Then
// |ph + c - d scale| < 2^-45 d scale < 2^-23 while d scale < 2^22, the FP64
// rule's two roundings move its t by at most 2^-52 t < 2^-30 from d scale, and
// r = (ph - floor(ph)) + c carries one more rounding (< 2^-23). So when r lies
// farther than 2^-20 from every integer, floor(t) = floor(ph) + floor(r); next
// to an integer (t at or near a grid boundary, d = 0), or out of range or not
// finite, the FP64 rule is evaluated as written. Integers below 2^22 are exact
// in FP32.
struct GridAxis {
    double lo, scale;
    float lo32, sh, sl;
    bool fast;   // lo is an FP32 value (the minimum of FP32 coordinates) and the split is finite
};

__device__ __forceinline__ GridAxis grid_axis(double lo, double scale) {
    GridAxis g;
    g.lo = lo;
    g.scale = scale;
    g.lo32 = __double2float_rn(lo);
    g.sh = __double2float_rn(scale);
    g.sl = __double2float_rn(__dsub_rn(scale, (double)g.sh));
    g.fast = (double)g.lo32 == lo && isfinite(g.sh) && isfinite(g.sl);
    return g;
}

__device__ __forceinline__ uint32_t grid_coord_fast(float v, const GridAxis &g) {
    if (g.fast) {
        const float b = -g.lo32;
        const float dh = __fadd_rn(v, b);
        const float bb = __fsub_rn(dh, v);
        const float dl = __fadd_rn(__fsub_rn(v, __fsub_rn(dh, bb)), __fsub_rn(b, bb));
        const float ph = __fmul_rn(dh, g.sh);
        const float pl = __fmaf_rn(dh, g.sh, -ph);
        const float c = __fmaf_rn(dh, g.sl, __fmaf_rn(dl, g.sh, pl));
        if (ph >= 0.f && ph < 4194304.f) {
            const float f = floorf(ph);
            const float r = __fadd_rn(__fsub_rn(ph, f), c);
            constexpr float M = 9.5367431640625e-07f;   // 2^-20
            float q = -2.f;
            if (r > M && r < 1.f - M) q = f;
            else if (r > 1.f + M && r < 2.f - M) q = f + 1.f;
            else if (r > M - 1.f && r < -M) q = f - 1.f;
            if (q >= 0.f) return q >= 2097151.f ? 2097151u : (uint32_t)q;
        }
    }
    return grid_coord(v, g.lo, g.scale);
}

// Lanes of the warp with this lane's digit, among those with ok (the others get
// nothing useful): one ballot a bit (the ranking rounds with __match_any_sync: a
// pass over 2^24 elements 260 us, 233 so).
__device__ __forceinline__ unsigned match_digit(unsigned d, bool ok) {
    unsigned m = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < kSortBits; b++) {
        const bool one = (d >> b) & 1u;
        const unsigned v = __ballot_sync(0xffffffffu, one);
        m &= one ? v : ~v;
    }
    return m;
}

// Digit counts of one key into the block's [passes][kSortBins] counters. (The high
// digits of a centrally concentrated system hold few values; shared-memory adds
// of a whole warp to one counter still beat finding the lanes that agree: build of
// 2^24 stars 3.40 ms, 3.60 with the four high digits added once per value.)
template <int PASSES>
__device__ __forceinline__ void count_digits(uint64_t k, int *h) {
#pragma unroll
    for (int p = 0; p < PASSES; p++) atomicAdd(&h[p * kSortBins + ((int)(k >> (p * kSortBits)) & (kSortBins - 1))], 1);
}

// Blocks (bx, m): member m's stars with member m's bounding cube. Each star's
// (x, y, z, m) is also packed into one float4 (caller order), so that the
// gather into key order reads one 16-byte record per star instead of four
// scattered 4-byte values (each costing a 32-byte sector). The digit counts of
// all sort passes are taken here, where the keys are in registers (the sort
// then reads them only to move them), and the first pass's look-back words are cleared.
__global__ void __launch_bounds__(256) keys_k(int64_t n, const int64_t *moff, int bpm, const float *x, const float *y,
                                              const float *z, const float *mass, const double *mbounds, uint64_t *key,
                                              float4 *xyzm, unsigned *ghist, uint4 *words, int64_t nwords4) {
    __shared__ int h[kKeyPasses * kSortBins];
    for (int b = threadIdx.x; b < kKeyPasses * kSortBins; b += 256) h[b] = 0;
    const int64_t nthr = (int64_t)gridDim.x * gridDim.y * 256;
    for (int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 256 + threadIdx.x; i < nwords4; i += nthr)
        words[i] = make_uint4(0, 0, 0, 0);
    const int m = blockIdx.y;
    const double sc = mbounds[5 * m + 4];
    const GridAxis gx = grid_axis(mbounds[5 * m], sc), gy = grid_axis(mbounds[5 * m + 1], sc),
                   gz = grid_axis(mbounds[5 * m + 2], sc);
    const int64_t s = max(moff[m], (int64_t)0), e = min(moff[m + 1], n);
    __syncthreads();
    for (int64_t i = s + (int64_t)blockIdx.x * 256 + threadIdx.x; i < e; i += (int64_t)bpm * 256) {
        const float xi = x[i], yi = y[i], zi = z[i];
        const uint64_t k = spread3(grid_coord_fast(xi, gx)) | (spread3(grid_coord_fast(yi, gy)) << 1) |
                           (spread3(grid_coord_fast(zi, gz)) << 2);
        key[i] = k;
        xyzm[i] = make_float4(xi, yi, zi, mass[i]);
        count_digits<kKeyPasses>(k, h);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kKeyPasses * kSortBins; b += 256)
        if (h[b]) atomicAdd(&ghist[b], (unsigned)h[b]);
}

// ---------------------------------------------------------------------------
// stable LSD radix sort of (key, index), 9-bit digits, one kernel a pass
// ---------------------------------------------------------------------------
// The digit counts of `passes` passes of a key array (sorts other than the build's).
__global__ void __launch_bounds__(256) sort_hist_k(int64_t n, const uint64_t *key, int passes, unsigned *ghist) {
    __shared__ int h[4 * kSortBins];
    for (int b = threadIdx.x; b < 4 * kSortBins; b += 256) h[b] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        count_digits<4>(key[i], h);
    __syncthreads();
    for (int b = threadIdx.x; b < passes * kSortBins; b += 256)
        if (h[b]) atomicAdd(&ghist[b], (unsigned)h[b]);
}

// One pass: the digit of element j is 9 key bits from `shift`, or (moff: the
// member pass) the member of its caller index, which groups the members while
// keeping each one's order. A block takes the next tile of TILE = 256 ITEMS
// elements. Each warp ranks its consecutive keys in ITEMS rounds of 32
// (warp-private digit counters), so the in-tile order is (warp, round, lane) =
// input order and the sort is stable; thread t owns digits 2t and 2t + 1,
// publishes their counts in the tile, and looks back for the counts before it
// (the words of tile t: words[t][kSortBins]); the tile is staged in shared
// memory in digit order and written out from there, consecutive threads to
// consecutive slots of a digit's output run. The digits' first slots are the
// exclusive scan of the digit counts `ghist` (or the members' offsets). The last
// pass also gathers the stars (pos). words_next: the next pass's words, cleared
// here tile by tile (null: none).
//
// One launch a pass and 24 B an element, against five launches and 32 B for a
// count, a three-kernel scan and a move: seven passes 190 -> 73 us on 100003
// stars, where launches and latency count. Large sorts are bound by the ranking
// rounds and the short output runs (512 digits a tile of 4096: 8 elements a run;
// 2^24 elements 233 us a pass, 1.7 TB/s).
template <int ITEMS>
struct SortSmem {
    unsigned short cnt[kSortThreads / 32][kSortBins];
    int gbase[kSortBins];                        // first output slot of each digit for this tile
    int lstart[kSortBins];                       // first staged slot of each digit
    uint64_t key[kSortThreads * ITEMS];
    int idx[kSortThreads * ITEMS];
    unsigned short dig[kSortThreads * ITEMS];
    int sw[kSortThreads / 32];
    int tile;
};

template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads) sort_pass_k(int64_t n, const uint64_t *key_in, const int *idx_in,
                                                            int shift, const int64_t *moff, int M,
                                                            const unsigned *ghist, int *ticket, unsigned *gave_up,
                                                            LbWait wait, unsigned *words, unsigned *words_next,
                                                            uint64_t *key_out, int *idx_out, const float4 *xyzm,
                                                            float4 *pos, DevState *st) {
    constexpr int NW = kSortThreads / 32, TILE = kSortThreads * ITEMS;
    static_assert(kSortBins == 2 * kSortThreads, "a thread owns two digits");
    extern __shared__ __align__(16) char sort_smem[];
    SortSmem<ITEMS> &S = *reinterpret_cast<SortSmem<ITEMS> *>(sort_smem);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        const int t = atomicAdd(ticket, 1);
        S.tile = lb_load(gave_up) ? -1 : t;
    }
    for (int b = lane; b < kSortBins / 2; b += 32) reinterpret_cast<unsigned *>(S.cnt[wid])[b] = 0;
    __syncthreads();
    const int tile = S.tile;
    if (tile < 0) return;   // a pass before left slots unwritten: its indices must not be used
    const int64_t tile0 = (int64_t)tile * TILE;
    const int64_t base = tile0 + wid * (32 * ITEMS);
    const int d0 = 2 * threadIdx.x;   // this thread's digits
    if (words_next) *reinterpret_cast<uint2 *>(words_next + (int64_t)tile * kSortBins + d0) = make_uint2(0, 0);
    uint64_t kk[ITEMS];
    int ix[ITEMS], digit[ITEMS], rank[ITEMS];
    // every load of the tile first, so that their latencies overlap (the
    // ranking rounds below synchronise the warp)
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int64_t j = base + r * 32 + lane;
        const bool ok = j < n;
        kk[r] = ok ? key_in[j] : 0ull;
        ix[r] = ok ? (idx_in ? idx_in[j] : (int)j) : 0;
    }
    // the digits' counts in the whole input (the member pass: the members' offsets)
    int g0 = 0, g1 = 0;
    if (!moff) {
        g0 = (int)__ldg(ghist + d0);
        g1 = (int)__ldg(ghist + d0 + 1);
    }
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int64_t j = base + r * 32 + lane;
        int d = kSortBins;
        if (j < n) d = moff ? member_of(moff, M, (int64_t)ix[r]) : (int)((kk[r] >> shift) & (kSortBins - 1));
        digit[r] = d;
        const unsigned peers = match_digit(d, d < kSortBins);
        int before = (d < kSortBins) ? S.cnt[wid][d] : 0;
        rank[r] = before + __popc(peers & lanemask_lt());
        __syncwarp();
        if (d < kSortBins && lane == __ffs(peers) - 1) S.cnt[wid][d] = (unsigned short)(before + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // per digit: the warps' counts become offsets within the digit's run of this tile
    int tot0 = 0, tot1 = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) {
        ushort2 *q = reinterpret_cast<ushort2 *>(&S.cnt[w][d0]);
        const ushort2 t = *q;
        *q = make_ushort2((unsigned short)tot0, (unsigned short)tot1);
        tot0 += t.x;
        tot1 += t.y;
    }
    unsigned *mine = words + (int64_t)tile * kSortBins + d0;
    const unsigned state = tile ? kLbSum : kLbPrefix;
    if (tile != wait.hold) {
        lb_store(mine, state | (unsigned)tot0);
        lb_store(mine + 1, state | (unsigned)tot1);
    }
    // digit runs in digit order: exclusive scans of the tile's totals and of the whole input's
    int total;
    const int ex = block_exclusive_scan<kSortThreads>(tot0 + tot1, S.sw, total);
    S.lstart[d0] = ex;
    S.lstart[d0 + 1] = ex + tot0;
    int first0, first1;
    if (moff) {
        first0 = d0 < M ? (int)moff[d0] : 0;
        first1 = d0 + 1 < M ? (int)moff[d0 + 1] : 0;
    } else {
        const int gx = block_exclusive_scan<kSortThreads>(g0 + g1, S.sw, total);
        first0 = gx;
        first1 = gx + g0;
    }
    // counts of this thread's digits in the tiles before, four tiles' words in flight
    bool fail = false;
    unsigned b0 = 0, b1 = 0;
    bool done0 = tile == 0, done1 = tile == 0;
    for (int t = tile - 1, spin = 0; !(done0 && done1);) {
        uint2 w[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const unsigned *p = words + (int64_t)max(t - q, 0) * kSortBins + d0;
            w[q].x = lb_load(p);
            w[q].y = lb_load(p + 1);
        }
        int used = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            // in order, while every tile so far was there (tile 0's words are prefixes)
            if (used == q && (done0 || (w[q].x >> 30)) && (done1 || (w[q].y >> 30))) {
                used = q + 1;
                if (!done0) {
                    b0 += w[q].x & kLbCount;
                    done0 = (w[q].x & kLbPrefix) != 0;
                }
                if (!done1) {
                    b1 += w[q].y & kLbCount;
                    done1 = (w[q].y & kLbPrefix) != 0;
                }
            }
        }
        t -= used;
        if (used == 0 && ++spin > wait.polls) {
            fail = true;
            break;
        }
    }
    if (tile && !fail) {
        lb_store(mine, kLbPrefix | ((b0 + (unsigned)tot0) & kLbCount));
        lb_store(mine + 1, kLbPrefix | ((b1 + (unsigned)tot1) & kLbCount));
    }
    S.gbase[d0] = first0 + (int)b0 - ex;
    S.gbase[d0 + 1] = first1 + (int)b1 - (ex + tot0);
    if (__syncthreads_or(fail)) {   // a wait gave up: nothing is written
        if (threadIdx.x == 0) {
            latch_err(st, kErrLookback);
            lb_store(gave_up, 1u);
        }
        return;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int64_t j = base + r * 32 + lane;
        if (j < n) {
            const int d = digit[r];
            const int slot = S.lstart[d] + S.cnt[wid][d] + rank[r];
            S.key[slot] = kk[r];
            S.idx[slot] = ix[r];
            S.dig[slot] = (unsigned short)d;
        }
    }
    __syncthreads();
    const int tn = (int)min((int64_t)TILE, n - tile0);
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int t = r * kSortThreads + threadIdx.x;
        if (t >= tn) break;
        const int64_t dst = (int64_t)S.gbase[S.dig[t]] + t;
        const int i = S.idx[t];
        key_out[dst] = S.key[t];
        idx_out[dst] = i;
        if (pos) pos[dst] = __ldg(&xyzm[i]);
    }
}

// Items a thread (tile / 256): small sorts in small tiles (more blocks), large
// ones in large tiles (longer output runs). Whole build in us with tiles of
// 1024, 2048, 4096: 195, 189, 203 on 200001 stars, 300, 272, 261 on 2^19,
// 473, 417, 387 on 2^20; 2^24: 3876 at 2048, 3820 at 4096.
constexpr int64_t kSortN4 = 1 << 17, kSortN8 = 1 << 18;
static int sort_items(int64_t n) { return n < kSortN4 ? 4 : n < kSortN8 ? 8 : 16; }

int64_t sort_words(int64_t n_max) {
    int64_t tiles = 1;
    for (int64_t n : {std::min(n_max, kSortN4 - 1), std::min(n_max, kSortN8 - 1), n_max})
        tiles = std::max<int64_t>(tiles, ceil_div(n, kSortThreads * sort_items(n)));
    return tiles * kSortBins;
}

template <int ITEMS>
static void sort_pass(rv_ctx *c, int64_t n, const uint64_t *ki, const int *ii, int shift, const int64_t *moff,
                      const unsigned *ghist, int *ticket, LbWait wait, unsigned *words, unsigned *next, uint64_t *ko,
                      int *io, const float4 *xyzm, float4 *pos, cudaStream_t s) {
    auto kern = sort_pass_k<ITEMS>;
    if (sizeof(SortSmem<ITEMS>) > 48 * 1024)
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem<ITEMS>));
    kern<<<ceil_div(n, kSortThreads * ITEMS), kSortThreads, sizeof(SortSmem<ITEMS>), s>>>(
        n, ki, ii, shift, moff, c->n_members, ghist, ticket, c->w.lb + kLbGaveUp, wait, words, next, ko, io, xyzm, pos,
        c->w.st);
    count_launch(c);
}

// Sorts key_a with identity indices; `counted`: the digit counts, tickets and
// the first pass's words are set up already (the build's first kernels). With
// pos, the stars xyzm are gathered into key order by the last pass.
rv_status radix_sort(rv_ctx *c, int64_t n, int passes, uint64_t **keys, int **idx, cudaStream_t s, bool member_pass,
                     bool counted, const float4 *xyzm, float4 *pos) {
    if (n <= 0) return RV_OK;
    Workspace &w = c->w;
    const int items = sort_items(n);
    unsigned *ghist = w.lb + kLbHist;
    int *tickets = reinterpret_cast<int *>(w.lb + kLbTickets);
    if (!counted) {
        const int ntiles = ceil_div(n, kSortThreads * items);
        rv_status r = cuda_check(c, cudaMemsetAsync(w.lb, 0, sizeof(unsigned) * kLbScan, s), "radix sort");
        if (r == RV_OK)
            r = cuda_check(c, cudaMemsetAsync(w.words[0], 0, sizeof(unsigned) * kSortBins * (size_t)ntiles, s), "radix sort");
        if (r != RV_OK) return r;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 1024), (int64_t)c->num_sms * 4));
        sort_hist_k<<<grid, 256, 0, s>>>(n, w.key_a, passes, ghist);
        count_launch(c);
    }
    uint64_t *kin = w.key_a, *kout = w.key_b;
    int *iin = nullptr, *iout = w.idx_b;
    const int total = passes + ((member_pass && c->n_members > 1) ? 1 : 0);
    for (int p = 0; p < total; p++) {
        const bool mem = p == passes, lastp = p + 1 == total;
        auto run = items == 4 ? sort_pass<4> : items == 8 ? sort_pass<8> : sort_pass<16>;
        run(c, n, kin, iin, p * kSortBits, mem ? w.moff : nullptr, mem ? nullptr : ghist + p * kSortBins, tickets + p,
            lb_wait(c, kLbStageSort + p), w.words[p & 1], lastp ? nullptr : w.words[(p + 1) & 1], kout, iout, lastp ? xyzm : nullptr,
            lastp ? pos : nullptr, s);
        // next pass reads what this one wrote
        uint64_t *tk = kin; kin = kout; kout = tk;
        int *ti = (iin == nullptr) ? w.idx_a : iin;
        iin = iout; iout = ti;
    }
    *keys = kin;
    *idx = iin;
    return cuda_check(c, cudaGetLastError(), "radix sort");
}

// ---------------------------------------------------------------------------
// small builds: bounding cube, keys, sort and gather of one system of up to
// kSmallSort stars in one block, the keys in shared memory over the seven passes
// (one tile, so a pass needs no look-back). The nine launches of the general path
// are mostly latency: build of 1000 stars 104 -> 58 us, of 4096 117 -> 87; at
// 8192 one SM's rate is what counts (130 against 124 us). The keys, their order
// and the cube are the same bits.
// ---------------------------------------------------------------------------
constexpr int64_t kSmallSort = 4096;
constexpr int kSmallThreads = 512, kSmallWarps = kSmallThreads / 32;

struct SmallArgs {
    int n;
    const int64_t *moff;
    const float *x, *y, *z, *mass;
    double *mbounds;
    int *mroot;
    unsigned *zero;   // the words later kernels count in
    int64_t nzero;
    uint64_t *key_out;
    int *perm;
    float4 *pos;
    DevState *st;
};

template <int ITEMS>
struct SmallSmem {
    uint64_t key[2][kSmallThreads * ITEMS];
    unsigned short idx[2][kSmallThreads * ITEMS];
    unsigned short cnt[kSmallWarps][kSortBins];
    int lstart[kSortBins];
    int sw[32];
    float red[6][kSmallWarps];
    double bounds[5];
};

template <int ITEMS>
__global__ void __launch_bounds__(kSmallThreads) small_sort_k(SmallArgs A) {
    extern __shared__ __align__(16) char small_smem[];
    SmallSmem<ITEMS> &S = *reinterpret_cast<SmallSmem<ITEMS> *>(small_smem);
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, n = A.n;
    for (int64_t i = t; i < A.nzero; i += kSmallThreads) A.zero[i] = 0;
    if (!offsets_fit(A.moff, 1, n) && t == 0) {
        latch_err(A.st, kErrOffsets);
        A.zero[kLbGaveUp] = 1;
    }
    // element r of a thread: the warp's consecutive elements in rounds of 32
    const int base = wid * (32 * ITEMS) + lane;
    float px[ITEMS], py[ITEMS], pz[ITEMS];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = base + r * 32;
        if (i < n) {
            px[r] = A.x[i];
            py[r] = A.y[i];
            pz[r] = A.z[i];
        }
    }
#pragma unroll
    for (int r = 0; r < ITEMS; r++)
        if (base + r * 32 < n) {
            lo[0] = fminf(lo[0], px[r]); hi[0] = fmaxf(hi[0], px[r]);
            lo[1] = fminf(lo[1], py[r]); hi[1] = fmaxf(hi[1], py[r]);
            lo[2] = fminf(lo[2], pz[r]); hi[2] = fmaxf(hi[2], pz[r]);
        }
    auto warp_minmax = [&]() {
#pragma unroll
        for (int a = 0; a < 3; a++)
            for (int o = 16; o > 0; o >>= 1) {
                lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
                hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
            }
    };
    warp_minmax();
    if (lane == 0)
        for (int a = 0; a < 3; a++) {
            S.red[a][wid] = lo[a];
            S.red[3 + a][wid] = hi[a];
        }
    __syncthreads();
    if (wid == 0) {
        for (int a = 0; a < 3; a++) {
            lo[a] = S.red[a][lane % kSmallWarps];
            hi[a] = S.red[3 + a][lane % kSmallWarps];
        }
        warp_minmax();
        if (lane == 0) {
            cube_of(lo, hi, S.bounds);
            for (int k = 0; k < 5; k++) A.mbounds[k] = A.st->bounds[k] = S.bounds[k];
            A.mroot[0] = -1;
            A.st->ncell = A.st->ngroup = 0;
        }
    }
    __syncthreads();
    const GridAxis gx = grid_axis(S.bounds[0], S.bounds[4]), gy = grid_axis(S.bounds[1], S.bounds[4]),
                   gz = grid_axis(S.bounds[2], S.bounds[4]);
    uint64_t kk[ITEMS];
    unsigned short ix[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = base + r * 32;
        kk[r] = i < n ? spread3(grid_coord_fast(px[r], gx)) | (spread3(grid_coord_fast(py[r], gy)) << 1) |
                            (spread3(grid_coord_fast(pz[r], gz)) << 2)
                      : 0ull;
        ix[r] = (unsigned short)i;
    }
    for (int p = 0; p < kKeyPasses; p++) {
        for (int b = lane; b < kSortBins / 2; b += 32) reinterpret_cast<unsigned *>(S.cnt[wid])[b] = 0;
        if (p > 0) {
#pragma unroll
            for (int r = 0; r < ITEMS; r++) {
                const int i = base + r * 32;
                if (i < n) {
                    kk[r] = S.key[p & 1][i];
                    ix[r] = S.idx[p & 1][i];
                }
            }
        }
        __syncwarp();
        unsigned short rank[ITEMS];
#pragma unroll
        for (int r = 0; r < ITEMS; r++) {
            const bool ok = base + r * 32 < n;
            const int d = ok ? (int)(kk[r] >> (p * kSortBits)) & (kSortBins - 1) : kSortBins;
            const unsigned peers = match_digit(d, ok);
            const int before = ok ? S.cnt[wid][d] : 0;
            rank[r] = (unsigned short)(before + __popc(peers & lanemask_lt()));
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1) S.cnt[wid][d] = (unsigned short)(before + __popc(peers));
            __syncwarp();
        }
        __syncthreads();
        // digits 2t, 2t + 1 (t < 256), two 16-bit counts a word (they stay below 2^16
        // together): the warps' counts become offsets in the runs; then the runs' starts
        unsigned tot = 0;
        if (t < kSortBins / 2) {
            unsigned v[kSmallWarps];
#pragma unroll
            for (int w = 0; w < kSmallWarps; w++) v[w] = reinterpret_cast<unsigned *>(S.cnt[w])[t];
#pragma unroll
            for (int w = 0; w < kSmallWarps; w++) {
                reinterpret_cast<unsigned *>(S.cnt[w])[t] = tot;
                tot += v[w];
            }
        }
        int total;
        const int t0 = (int)(tot & 0xffffu), ex = block_exclusive_scan<kSmallThreads>(t0 + (int)(tot >> 16), S.sw, total);
        if (t < kSortBins / 2) {
            S.lstart[2 * t] = ex;
            S.lstart[2 * t + 1] = ex + t0;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ITEMS; r++)
            if (base + r * 32 < n) {
                const int d = (int)(kk[r] >> (p * kSortBits)) & (kSortBins - 1);
                const int slot = S.lstart[d] + S.cnt[wid][d] + rank[r];
                S.key[(p + 1) & 1][slot] = kk[r];
                S.idx[(p + 1) & 1][slot] = ix[r];
            }
        __syncthreads();
    }
    constexpr int last = kKeyPasses & 1;
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
        const int i = r * kSmallThreads + t;
        if (i < n) {
            const int j = S.idx[last][i];
            A.key_out[i] = S.key[last][i];
            A.perm[i] = j;
            A.pos[i] = make_float4(A.x[j], A.y[j], A.z[j], A.mass[j]);
        }
    }
}

template <int ITEMS>
static rv_status small_sort(rv_ctx *c, const SmallArgs &A, cudaStream_t s) {
    auto kern = small_sort_k<ITEMS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem<ITEMS>));
    if (e != cudaSuccess) return cuda_check(c, e, "small sort");
    kern<<<1, kSmallThreads, sizeof(SmallSmem<ITEMS>), s>>>(A);
    count_launch(c);
    return cuda_check(c, cudaGetLastError(), "small sort");
}

// ---------------------------------------------------------------------------
// topology
// ---------------------------------------------------------------------------
__device__ __forceinline__ int diff_level(uint64_t a, uint64_t b) {
    uint64_t d = a ^ b;
    if (d == 0) return kLevels;  // equal keys never separate
    int h = 63 - __clzll((long long)d);
    return (65 - h) / 3;
}

// Window of D values for one block: D(j) for j in [b0 - n_leaf + 1, b0 + NT + n_leaf].
// Out-of-range positions are not boundaries (99); D(0) = D(n) = 0.
// A member's first star is a cut at every level, like position 0.
__device__ void load_window(int64_t n, const uint64_t *key, int64_t b0, int n_leaf, const int64_t *moff, int M,
                            unsigned char *win) {
    int wlen = kTopoBlock + 2 * n_leaf;
    for (int t = threadIdx.x; t < wlen; t += blockDim.x) {
        int64_t j = b0 - n_leaf + 1 + t;
        int d;
        if (j < 0 || j > n) d = 99;
        else if (j == 0 || j == n) d = 0;
        else if (M > 1 && moff[member_of(moff, M, j)] == j) d = 0;
        else d = diff_level(key[j - 1], key[j]);
        win[t] = (unsigned char)d;
    }
}

// lambda_i from the window (i = b0 + threadIdx.x): the smallest level l such
// that positions b1 <= i < b2, b2 - b1 <= n_leaf, are both cuts at l.
__device__ __forceinline__ int leaf_level(const unsigned char *win, int t, int n_leaf) {
    // win index of position j is j - (b0 - n_leaf + 1); i sits at t + n_leaf - 1
    const int wi = t + n_leaf - 1;
    int pm = 99, L = 99;
    for (int s = n_leaf - 1; s >= 0; s--) {
        int u = n_leaf - s;
        pm = min(pm, (int)win[wi + u]);
        L = min(L, max((int)win[wi - s], pm));
    }
    return min(L, kMaxLevel);
}

// Per-level ballots of "a cell starts at star i at level l" (D_i <= l <= lambda_i)
// and their warp prefix counts (shared, [kLevels][NW]).
struct TopoBallots {
    unsigned mask[kLevels];
};

__device__ __forceinline__ void topo_ballots(bool valid, int Di, int lam, TopoBallots &b) {
#pragma unroll
    for (int l = 0; l < kLevels; l++) b.mask[l] = __ballot_sync(0xffffffffu, valid && Di <= l && l <= lam);
}

__global__ void __launch_bounds__(kTopoBlock) topo_count_k(int64_t n, const uint64_t *key, int n_leaf,
                                                           const int64_t *moff, int M, uint8_t *dlev,
                                                           uint8_t *lam_out, int *lvcnt, int nblk) {
    extern __shared__ unsigned char win[];
    __shared__ int wc[kLevels][kTopoBlock / 32];
    int64_t b0 = (int64_t)blockIdx.x * kTopoBlock;
    load_window(n, key, b0, n_leaf, moff, M, win);
    __syncthreads();
    int64_t i = b0 + threadIdx.x;
    bool valid = i < n;
    int Di = 0, lam = -1;
    if (valid) {
        Di = win[threadIdx.x + n_leaf - 1];
        lam = leaf_level(win, threadIdx.x, n_leaf);
        dlev[i] = (uint8_t)Di;
        lam_out[i] = (uint8_t)lam;
    }
    TopoBallots b;
    topo_ballots(valid, Di, lam, b);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0)
        for (int l = 0; l < kLevels; l++) wc[l][wid] = __popc(b.mask[l]);
    __syncthreads();
    if (threadIdx.x < kLevels) {
        int s = 0;
        for (int w = 0; w < kTopoBlock / 32; w++) s += wc[threadIdx.x][w];
        lvcnt[(int64_t)threadIdx.x * nblk + blockIdx.x] = s;
    }
}

__device__ __forceinline__ int4 cell_box(uint64_t key, int l) {
    int sh = 3 * (kMaxLevel - l);
    uint64_t pre = (sh >= 64) ? 0ull : ((key >> sh) << sh);
    return make_int4((int)compact3(pre), (int)compact3(pre >> 1), (int)compact3(pre >> 2), l);
}

// Writes every cell's box, first star, child first, parent; and, as the star
// that ends a cell, its end star and child end.
__global__ void __launch_bounds__(kTopoBlock) topo_write_k(int64_t n, const uint64_t *key, const uint8_t *dlev,
                                                           const uint8_t *lamv, const int *lvscan, int nblk,
                                                           int64_t cap, const int64_t *moff, int M, int4 *cbox,
                                                           int *clink, int *cparent, int *carrive, int *mroot,
                                                           DevState *st) {
    __shared__ int wp[kLevels][kTopoBlock / 32];
    __shared__ int lvoff[kLevels + 1];
    __shared__ int bbase[kLevels + 1];
    if (st->ncell <= 0) return;   // the sort or the scan gave up: no counts to place cells by
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t i = (int64_t)blockIdx.x * kTopoBlock + threadIdx.x;
    bool valid = i < n;
    int Di = valid ? dlev[i] : 0, lam = valid ? lamv[i] : -1;
    TopoBallots b;
    topo_ballots(valid, Di, lam, b);
    if (lane == 0)
        for (int l = 0; l < kLevels; l++) wp[l][wid] = __popc(b.mask[l]);
    if (threadIdx.x <= kLevels) {
        int l = threadIdx.x;
        // level offsets: scanned value at the first block of each level; total at the end
        int tot = st->ncell;
        lvoff[l] = (l < kLevels) ? lvscan[(int64_t)l * nblk] : tot;
        bbase[l] = (l < kLevels) ? lvscan[(int64_t)l * nblk + blockIdx.x] : tot;
    }
    __syncthreads();
    if (threadIdx.x < kLevels) {
        int run = 0;
        for (int w = 0; w < kTopoBlock / 32; w++) {
            int t = wp[threadIdx.x][w];
            wp[threadIdx.x][w] = run;
            run += t;
        }
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x <= kLevels) st->lvoff[threadIdx.x] = lvoff[threadIdx.x];
    if (!valid) return;
    const unsigned lt = lanemask_lt();
    auto outside = [&](int c) -> bool { return c < 0 || c >= cap; };
    // exclusive global rank of star i among cells of level l
    auto rank = [&](int l) -> int { return bbase[l] + wp[l][wid] + __popc(b.mask[l] & lt); };
    uint64_t k = key[i];
    for (int l = Di; l <= lam; l++) {
        int c = rank(l);
        if (outside(c)) { latch_err(st, kErrCells); return; }
        cbox[c] = cell_box(k, l);
        clink[4 * c + 0] = (l < lam) ? rank(l + 1) : 0;  // first child: cell (l + 1, i)
        if (l == lam) clink[4 * c + 1] = 0;
        clink[4 * c + 2] = (int)i;
        cparent[c] = (l == 0) ? -1 : rank(l - 1) - ((Di == l) ? 1 : 0);
        carrive[c] = 0;
        if (l == 0) mroot[member_of(moff, M, i)] = c;
    }
    // cells containing star i-1 that end at i: levels D(i)..lambda_{i-1}
    if (i > 0) {
        int lp = lamv[i - 1];
        for (int l = Di; l <= lp; l++) {
            int c = rank(l) - 1;
            if (outside(c)) { latch_err(st, kErrCells); return; }
            clink[4 * c + 3] = (int)i;
            if (l < lp) clink[4 * c + 1] = rank(l + 1);
        }
    }
    // the last cell of every level that holds star n-1 ends at n
    if (i == n - 1) {
        for (int l = 0; l <= lam; l++) {
            int c = lvoff[l + 1] - 1;
            if (outside(c)) { latch_err(st, kErrCells); return; }
            clink[4 * c + 3] = (int)n;
            if (l < lam) clink[4 * c + 1] = lvoff[l + 2];
        }
    }
}

// ---------------------------------------------------------------------------
// walk groups
// ---------------------------------------------------------------------------
// A unit is a maximal cell with at most U = 16 G stars (one with <= U stars
// whose parent has more, or a member's root) or a leaf with more than U stars.
// Each unit is cut into runs of G consecutive stars in key order, the last run
// possibly shorter; each run is a group. A group's box is the tightest box on
// the member's integer grid that holds its stars' grid cells: per axis
// [min q, max q + 1), q the star's de-interleaved key. Every star lies in its
// group's box, so a cell the box-box test accepts passes the opening test for
// each star of the group.
//
// One pass over the cells in tiles of `tc` (<= 256) cells: a thread counts its
// cell's groups, the block scans the counts and looks back for the groups of
// the tiles before, and its warps take the tile's groups one by one. (A count, a
// three-kernel scan and a writing pass whose warps took a unit's groups in turn:
// 35 us on 100003 stars, hidden now behind the multipoles.)
struct GroupArgs {
    const uint64_t *skey;
    const int4 *cbox, *clink;
    const int *cparent;
    int G, U, tc;
    int64_t cap;
    unsigned *words;   // look-back words, zero before the launch
    int *ticket;
    LbWait wait;
    int4 *groups;
    int *garrive;
    DevState *st;
};

struct GroupSmem {
    int ofs[256], first[256], end[256];   // per cell of the tile: its first group, its stars
    int sw[8], tile;
    unsigned before;
    bool ok;
};

__device__ __forceinline__ int unit_groups(const GroupArgs &A, int c, int ncell, int4 &lk) {
    lk = A.clink[c];
    const int cnt = lk.w - lk.z;
    bool unit = false;
    if (cnt > A.U) {
        unit = (lk.x == lk.y);   // an overfull leaf
    } else if (A.cbox[c].w == 0) {
        unit = true;             // a member's root
    } else {
        const int p = A.cparent[c];
        if (p >= 0 && p < ncell) {
            const int4 pl = A.clink[p];
            unit = (pl.w - pl.z) > A.U;
        }
    }
    return unit ? (cnt + A.G - 1) / A.G : 0;
}

__device__ void write_groups(const GroupArgs &A, GroupSmem &S) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ncell = (int)min((int64_t)A.st->ncell, A.cap);
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) S.tile = atomicAdd(A.ticket, 1);
        __syncthreads();
        const int tile = S.tile, c0 = tile * A.tc;
        if (c0 >= ncell) return;
        const int c = c0 + threadIdx.x;
        int4 lk = make_int4(0, 0, 0, 0);
        int cnt = 0;
        if ((int)threadIdx.x < A.tc && c < ncell) cnt = unit_groups(A, c, ncell, lk);
        int total;
        const int ex = block_exclusive_scan<256>(cnt, S.sw, total);
        S.ofs[threadIdx.x] = ex;
        S.first[threadIdx.x] = lk.z;
        S.end[threadIdx.x] = lk.w;
        if (wid == 0) {
            if (lane == 0 && tile != A.wait.hold)
                lb_store(A.words + tile, (tile ? kLbSum : kLbPrefix) | (unsigned)total);
            unsigned before = 0;
            const bool ok = lb_sum_before(A.words, tile, A.wait.polls, before);
            if (lane == 0) {
                if (ok && tile) lb_store(A.words + tile, kLbPrefix | ((before + (unsigned)total) & kLbCount));
                if (!ok) latch_err(A.st, kErrLookback);
                lb_total(&A.st->ngroup, ok, c0 + A.tc >= ncell, (int)before + total);
                S.before = before;
                S.ok = ok;
            }
        }
        __syncthreads();
        if (!S.ok) return;
        for (int r = wid; r < total; r += 8) {
            int lo = 0, hi = A.tc - 1;   // group r's cell: the last one whose first group is at or before r
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (S.ofs[mid] <= r) lo = mid; else hi = mid - 1;
            }
            const int first = S.first[lo] + (r - S.ofs[lo]) * A.G;
            const int cnt = min(A.G, S.end[lo] - first);
            unsigned qlo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, qhi[3] = {0u, 0u, 0u};
            for (int i = lane; i < cnt; i += 32) {   // a run may hold up to 64 stars
                const uint64_t key = A.skey[first + i];
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    const unsigned q = compact3(key >> a);
                    qlo[a] = min(qlo[a], q);
                    qhi[a] = max(qhi[a], q + 1);
                }
            }
#pragma unroll
            for (int a = 0; a < 3; a++) {
                qlo[a] = __reduce_min_sync(0xffffffffu, qlo[a]);
                qhi[a] = __reduce_max_sync(0xffffffffu, qhi[a]);
            }
            if (lane == 0) {
                const int g = (int)S.before + r;
                A.groups[2 * g] = make_int4(first, cnt, (int)qlo[0], (int)qlo[1]);
                A.groups[2 * g + 1] = make_int4((int)qlo[2], (int)qhi[0], (int)qhi[1], (int)qhi[2]);
                A.garrive[g] = 0;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// multipoles, bottom-up: each leaf computes its moments from its stars; the
// last child to finish a parent (atomic arrival count) computes the parent
// from its children in child order, so the result does not depend on timing.
// FP32, accumulated relative to the cell's geometric centre.
// ---------------------------------------------------------------------------
// Moments are stored relative to the cell's geometric centre c0 (geo_centre):
// (M, com - c0), (Qxx, Qyy, Qzz, Qxy), (Qxz, Qyz, 0, 0).
struct Mom {
    float M, cx, cy, cz, q[6];  // cx..cz: centre of mass minus c0; q: xx, yy, zz, xy, xz, yz
};

__device__ __forceinline__ void store_mom(float4 *cmom, int c, const Mom &m) {
    cmom[3 * c + 0] = make_float4(m.M, m.cx, m.cy, m.cz);
    cmom[3 * c + 1] = make_float4(m.q[0], m.q[1], m.q[2], m.q[3]);
    cmom[3 * c + 2] = make_float4(m.q[4], m.q[5], 0.f, 0.f);
}



__device__ __forceinline__ void add_q(float q[6], float m, float dx, float dy, float dz) {
    float d2 = dx * dx + dy * dy + dz * dz;
    q[0] += m * (3.f * dx * dx - d2);
    q[1] += m * (3.f * dy * dy - d2);
    q[2] += m * (3.f * dz * dz - d2);
    q[3] += m * 3.f * dx * dy;
    q[4] += m * 3.f * dx * dz;
    q[5] += m * 3.f * dy * dz;
}

// One arrival at a cell: this thread's moments before it, the other children's
// moments after it (acquire and release in one operation).
__device__ __forceinline__ int arrive_acq_rel(int *p) {
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
    return old;
}

struct MomentArgs {
    int64_t n;
    const float4 *pos;
    const int4 *cbox, *clink;
    const int *cparent;
    int *carrive;
    float4 *cmom;
    int64_t cap;
    const int64_t *moff;
    int M;
    const double *mbounds;
    DevState *st;
};

// What bounds a small build is the chain from the deepest leaf to the root (10
// to 20 levels of a few dependent round trips each): there (BATCH 8) a leaf's
// stars and all of a cell's children are in flight at once and the parent's
// links are loaded beside the arrival. A large one is bound by the threads in
// flight, and takes them one by one (BATCH 1) in a third of the registers. The
// sums run in the same order either way: the moments are the same bits (80 us
// alone before on 100003 stars, 50 now). Blocks block, block + nblocks, ... of
// 256 cells.
template <int BATCH>
__device__ void climb_moments(const MomentArgs &A, int block, int nblocks) {
    const int ncell = (int)min((int64_t)A.st->ncell, A.cap);
    for (int c = block * 256 + threadIdx.x; c < ncell; c += nblocks * 256) {
        const int4 lk = A.clink[c];
        if (lk.y != lk.x) continue;  // not a leaf
        if (lk.z < 0 || lk.w > A.n || lk.z >= lk.w) { latch_err(A.st, kErrCells); continue; }
        const int mb = member_of(A.moff, A.M, lk.z);
        const float lo[3] = {(float)A.mbounds[5 * mb], (float)A.mbounds[5 * mb + 1], (float)A.mbounds[5 * mb + 2]};
        const float unit = (float)(A.mbounds[5 * mb + 3] / 2097152.0);
        float g[3];
        geo_centre(A.cbox[c], lo, unit, g);
        int par = A.cparent[c];
        Mom m = {};
        float sx = 0.f, sy = 0.f, sz = 0.f;
        auto stars = [&](auto &&take) {
            for (int j = lk.z; j < lk.w; j += BATCH) {
                float4 p[BATCH];
#pragma unroll
                for (int k = 0; k < BATCH; k++)
                    if (j + k < lk.w) p[k] = __ldg(&A.pos[j + k]);
#pragma unroll
                for (int k = 0; k < BATCH; k++)
                    if (j + k < lk.w) take(p[k]);
            }
        };
        stars([&](const float4 &p) {
            m.M += p.w;
            sx += p.w * (p.x - g[0]);
            sy += p.w * (p.y - g[1]);
            sz += p.w * (p.z - g[2]);
        });
        if (m.M > 0.f) {
            m.cx = sx / m.M; m.cy = sy / m.M; m.cz = sz / m.M;
            stars([&](const float4 &p) {
                add_q(m.q, p.w, (p.x - g[0]) - m.cx, (p.y - g[1]) - m.cy, (p.z - g[2]) - m.cz);
            });
        }
        store_mom(A.cmom, c, m);
        // climb while this thread is the last child to arrive (at most 21 levels)
        int cur = c;
        for (int guard = 0; guard <= kMaxLevel; guard++) {
            const int p = par;
            if (p < 0) break;
            if (p >= cur) { latch_err(A.st, kErrCells); break; }  // parents precede children
            const int4 pl = A.clink[p], pb = A.cbox[p];
            par = A.cparent[p];
            const int nch = pl.y - pl.x;
            if (pl.x <= p || pl.y > ncell || nch < 1 || nch > 8) { latch_err(A.st, kErrCells); break; }
            if (arrive_acq_rel(&A.carrive[p]) != nch - 1) break;
            float pg[3];
            geo_centre(pb, lo, unit, pg);
            Mom P = {};
            float px = 0.f, py = 0.f, pz = 0.f;
            auto first = [&](const float4 &a, const int4 &b) {
                float cg[3];
                geo_centre(b, lo, unit, cg);
                P.M += a.x;
                px += a.x * ((cg[0] - pg[0]) + a.y);
                py += a.x * ((cg[1] - pg[1]) + a.z);
                pz += a.x * ((cg[2] - pg[2]) + a.w);
            };
            auto second = [&](const float4 &a, const float4 &b, const float2 &e, const int4 &bx) {
                float cg[3];
                geo_centre(bx, lo, unit, cg);
                P.q[0] += b.x; P.q[1] += b.y; P.q[2] += b.z; P.q[3] += b.w; P.q[4] += e.x; P.q[5] += e.y;
                add_q(P.q, a.x, ((cg[0] - pg[0]) + a.y) - P.cx, ((cg[1] - pg[1]) + a.z) - P.cy,
                      ((cg[2] - pg[2]) + a.w) - P.cz);
            };
            auto load_a = [&](int ch) { return __ldcg(&A.cmom[3 * ch]); };
            auto load_b = [&](int ch) { return __ldcg(&A.cmom[3 * ch + 1]); };
            auto load_e = [&](int ch) { return __ldcg(reinterpret_cast<const float2 *>(&A.cmom[3 * ch + 2])); };
            if (BATCH == 8) {   // every record of the children at once
                float4 a[8], b[8];
                float2 e[8];
                int4 bx[8];
#pragma unroll
                for (int k = 0; k < 8; k++)
                    if (k < nch) {
                        a[k] = load_a(pl.x + k);
                        bx[k] = A.cbox[pl.x + k];
                        b[k] = load_b(pl.x + k);
                        e[k] = load_e(pl.x + k);
                    }
#pragma unroll
                for (int k = 0; k < 8; k++)
                    if (k < nch) first(a[k], bx[k]);
                if (P.M > 0.f) {
                    P.cx = px / P.M; P.cy = py / P.M; P.cz = pz / P.M;
#pragma unroll
                    for (int k = 0; k < 8; k++)
                        if (k < nch) second(a[k], b[k], e[k], bx[k]);
                }
            } else {
                for (int ch = pl.x; ch < pl.y; ch++) first(load_a(ch), A.cbox[ch]);
                if (P.M > 0.f) {
                    P.cx = px / P.M; P.cy = py / P.M; P.cz = pz / P.M;
                    for (int ch = pl.x; ch < pl.y; ch++) second(load_a(ch), load_b(ch), load_e(ch), A.cbox[ch]);
                }
            }
            store_mom(A.cmom, p, P);
            cur = p;
        }
    }
}

constexpr int64_t kLatencyBuild = 1 << 20;   // (2^19 stars: build 268 us against 273)

// Walk groups and multipoles need the topology alone and not one another: one
// launch, the first gblocks blocks write the groups while the others climb.
template <int BATCH>
__global__ void __launch_bounds__(256, BATCH == 8 ? 1 : 4) groups_moments_k(GroupArgs GA, MomentArgs MA, int gblocks) {
    __shared__ GroupSmem S;
    if ((int)blockIdx.x < gblocks) write_groups(GA, S);
    else climb_moments<BATCH>(MA, blockIdx.x - gblocks, gridDim.x - gblocks);
}

// ---------------------------------------------------------------------------
// driver
// ---------------------------------------------------------------------------
static int grid_for(rv_ctx *c, int64_t n, int per_block) {
    int64_t b = (n + per_block - 1) / per_block;
    int64_t cap = (int64_t)c->num_sms * 8;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, cap));
}

// Copies the member offsets to the device only when they differ from the
// last ones sent (a captured step must not copy from host memory).
rv_status upload_offsets(rv_ctx *c, int M, const int64_t *offsets, cudaStream_t s) {
    bool same = c->moff_on_device && c->n_members == M;
    for (int k = 0; k <= M && same; k++) same = (c->moff_host[k] == offsets[k]);
    if (same) return RV_OK;
    for (int k = 0; k <= M; k++) c->moff_host[k] = offsets[k];
    c->n_members = M;
    rv_status r = cuda_check(c, cudaMemcpyAsync(c->w.moff, c->moff_host, sizeof(int64_t) * (M + 1),
                                                cudaMemcpyHostToDevice, s), "member offsets");
    if (r == RV_OK) r = cuda_check(c, cudaStreamSynchronize(s), "member offsets");
    if (r == RV_OK) c->moff_on_device = true;
    return r;
}

// Members are independent systems stored one after another (offsets on the
// host, M >= 1). Each gets its own bounding cube, keys, tree and groups; all
// of them share these launches, and the walk serves them together.
rv_status build_tree(rv_ctx *c, int n_members, const int64_t *offsets, const float *x, const float *y,
                     const float *z, const float *m, cudaStream_t s) {
    Workspace &w = c->w;
    const int M = n_members;
    const int64_t n = offsets[M];
    c->n = n;
    c->built = false;
    int64_t big = 0;
    for (int k = 0; k < M; k++) big = std::max<int64_t>(big, offsets[k + 1] - offsets[k]);
    c->max_member = big;
    rv_status r = upload_offsets(c, M, offsets, s);
    if (r != RV_OK) return r;
    if (n == 0) {
        r = cuda_check(c, cudaMemsetAsync(w.st, 0, sizeof(DevState), s), "state reset");
        if (r == RV_OK) c->built = true;
        return r;
    }
    const int nblk = ceil_div(n, kTopoBlock);
    // what the build clears and launches follows its own stars, not the context's: cells of n
    // stars (at most 8 children of every split cell, of which a level has n / (n_leaf + 1))
    const int64_t cells = std::min<int64_t>(
        c->cell_cap, M + 2 + kMaxLevel * std::min<int64_t>(n, 8 * n / (c->cfg.n_leaf + 1) + 8));
    // cells a tile of the groups pass (few in small builds: more blocks); cleared
    // first: tickets, digit counts, the look-back words of the topology scan and of that pass
    const int tc = n < (1 << 19) ? 64 : 256;
    const int64_t lb_groups = kLbGroups(n), nzero = lb_groups + 2 + ceil_div(cells, tc);
    uint64_t *skey;
    int *perm;
    if (M == 1 && n <= kSmallSort) {
        skey = w.key_b;   // where the seven passes of a larger system end
        perm = w.idx_b;
        const SmallArgs A{(int)n, w.moff, x, y, z, m, w.mbounds, w.mroot, w.lb, nzero, skey, perm, w.pos, w.st};
        static_assert(kSmallSort <= 8 * kSmallThreads, "a thread's share");
        r = n <= 2 * kSmallThreads ? small_sort<2>(c, A, s) : small_sort<8>(c, A, s);
        if (r != RV_OK) return r;
    } else {
        // bounds and keys: blocks per member sized by the largest member
        const int bpm = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(big, kBoundsChunk), 512 / M + 1));
        bounds_k<<<dim3(bpm, M), 256, 0, s>>>(n, w.moff, bpm, x, y, z, w.bpart, w.barrive, w.mbounds, w.st, w.lb, nzero,
                                              w.mroot);
        count_launch(c);
        // (each block adds its digit counts to the global ones: at least 1024 stars a block)
        const int kpm = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(big, 1024), (int64_t)c->num_sms * 8 / M + 1));
        // the packed stars live in the group records' space until the gather: the
        // groups are written after it (32 B per star of room there, 16 needed)
        float4 *xyzm = reinterpret_cast<float4 *>(w.groups);
        const int64_t tiles = ceil_div(n, kSortThreads * sort_items(n));
        keys_k<<<dim3(kpm, M), 256, 0, s>>>(n, w.moff, kpm, x, y, z, m, w.mbounds, w.key_a, xyzm, w.lb + kLbHist,
                                            reinterpret_cast<uint4 *>(w.words[0]), tiles * kSortBins / 4);
        count_launch(c);
        if ((r = radix_sort(c, n, kKeyPasses, &skey, &perm, s, true, true, xyzm, w.pos)) != RV_OK) return r;
    }
    w.skey = skey;
    w.perm = perm;
    // topology
    size_t win = kTopoBlock + 2 * c->cfg.n_leaf;
    topo_count_k<<<nblk, kTopoBlock, win, s>>>(n, skey, c->cfg.n_leaf, w.moff, M, w.dlev, w.lam, w.lvcnt, nblk);
    count_launch(c);
    unsigned *lb = w.lb + kLbScan;   // cleared by bounds_k
    if ((r = scan_launch(c, w.lvcnt, (int64_t)kLevels * nblk, &w.st->ncell, lb + 1, reinterpret_cast<int *>(lb),
                         w.lb + kLbGaveUp, s)) != RV_OK)
        return r;
    topo_write_k<<<nblk, kTopoBlock, 0, s>>>(n, skey, w.dlev, w.lam, w.lvcnt, nblk, c->cell_cap, w.moff, M, w.cbox,
                                             w.clink, w.cparent, w.carrive, w.mroot, w.st);
    count_launch(c);
    // groups and multipoles
    const int4 *clink4 = reinterpret_cast<const int4 *>(w.clink);
    const int gblocks = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(cells, tc), c->num_sms));
    const int mblocks = grid_for(c, cells, 256);
    const GroupArgs GA{skey, w.cbox, clink4, w.cparent, c->cfg.group, 16 * c->cfg.group, tc, c->cell_cap,
                       w.lb + lb_groups + 1, reinterpret_cast<int *>(w.lb + lb_groups),
                       lb_wait(c, kLbStageGroups), w.groups, w.garrive, w.st};
    const MomentArgs MA{n, w.pos, w.cbox, clink4, w.cparent, w.carrive, w.cmom, c->cell_cap, w.moff, M, w.mbounds, w.st};
    // (one wave of latency-bound blocks as long as the cells fit it)
    if (n < kLatencyBuild) groups_moments_k<8><<<gblocks + mblocks, 256, 0, s>>>(GA, MA, gblocks);
    else groups_moments_k<1><<<gblocks + mblocks, 256, 0, s>>>(GA, MA, gblocks);
    count_launch(c);
    r = cuda_check(c, cudaGetLastError(), "build_tree");
    if (r == RV_OK) c->built = true;
    return r;
}

}  // namespace rv

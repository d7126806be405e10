// chain.cu -- the regularised chain's coupling to the tree (Sect. 2), the
// kick-drift-kick step and the FP64 energy/momentum totals.
//
// The chain (an SMBH, or an SMBH pair with the stars absorbed into it) is
// seen by the tree as one unsoftened particle at its centre of mass. Stars
// near it ("perturbers") get the pull of the resolved members instead of the
// centre-of-mass point mass; each member feels the perturbers directly; the
// centre-of-mass force is corrected by Eq. 3. All of this is unsoftened FP64;
// sums run in a fixed order so results do not depend on scheduling.
#include <cooperative_groups.h>

#include <algorithm>

#include "rv_internal.cuh"

namespace rv {

// ---------------------------------------------------------------------------
// perturber selection
// ---------------------------------------------------------------------------
// FP32 squared distance, every operation rounded separately in this order.
__device__ __forceinline__ float dist2_f32(float x, float y, float z, float cx, float cy, float cz) {
    float dx = __fsub_rn(x, cx), dy = __fsub_rn(y, cy), dz = __fsub_rn(z, cz);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

__device__ __forceinline__ float3 centre_of(const float *cdev, float3 chost) {
    return cdev ? make_float3(cdev[0], cdev[1], cdev[2]) : chost;
}

// Membership test of a sphere-like selection around a chain centre:
//   mode 1 (radius): d2 < r2 (FP32);
//   mode 3 (tidal criterion of Eq. 2): r < (2 m_j / (gamma M))^(1/3) r_crit,
//   taken without a cube root in FP64, one rounding per operation:
//   (d2 d2) d2 < (q q) rc6, q = (2 m_j) / (gamma M), rc6 = (rc2 rc2) rc2.
// M is the chain's FP32 total mass (the 4th value of its centre record).
struct SelRule {
    int mode;
    float r2;         // mode 1
    const float *m;   // mode 3: star masses
    float gamma;      // mode 3
    double rc6;       // mode 3
};

__device__ __forceinline__ bool sel_inside(const SelRule &R, float d2, int64_t i, float mchain) {
    if (R.mode != 3) return d2 < R.r2;
    const double dd = (double)d2;
    const double q = __ddiv_rn(__dmul_rn(2.0, (double)R.m[i]), __dmul_rn((double)R.gamma, (double)mchain));
    return __dmul_rn(__dmul_rn(dd, dd), dd) < __dmul_rn(__dmul_rn(q, q), R.rc6);
}

static SelRule sel_rule(int mode, float radius, const float *m, float gamma) {
    SelRule R;
    R.mode = mode;
    R.r2 = radius * radius;   // one FP32 product
    R.m = m;
    R.gamma = gamma;
    const double rc2 = (double)radius * (double)radius;
    R.rc6 = (rc2 * rc2) * rc2;
    return R;
}

// (it also clears the total that the scan after it adds up)
__global__ void sel_radius_flag_k(int64_t n, const float *x, const float *y, const float *z, const float *cdev,
                                  float4 chost, SelRule R, int *flag, int *total) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *total = 0;
    const float3 c = centre_of(cdev, make_float3(chost.x, chost.y, chost.z));
    const float mc = cdev ? cdev[3] : chost.w;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        flag[i] = sel_inside(R, dist2_f32(x[i], y[i], z[i], c.x, c.y, c.z), i, mc) ? 1 : 0;
}

__global__ void sel_radius_write_k(int64_t n, const float *x, const float *y, const float *z, const float *cdev,
                                   float4 chost, SelRule R, const int *ofs, const int *total, int cap, int *idx,
                                   int *count, DevState *st) {
    const int t = *total;
    if (t < 0) {   // the scan gave up: no offsets, so nothing is selected
        if (blockIdx.x == 0 && threadIdx.x == 0) *count = 0;
        return;
    }
    const float3 c = centre_of(cdev, make_float3(chost.x, chost.y, chost.z));
    const float mc = cdev ? cdev[3] : chost.w;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (sel_inside(R, dist2_f32(x[i], y[i], z[i], c.x, c.y, c.z), i, mc)) {
            int p = ofs[i];
            if (p < cap) idx[p] = (int)i;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *count = min(t, cap);
        if (t > cap) latch_err(st, kErrPert);
    }
}

// key = bits of the (non-negative) FP32 squared distance: integer order = float order
__global__ void sel_knn_keys_k(int64_t n, const float *x, const float *y, const float *z, const float *cdev,
                               float3 chost, uint64_t *key) {
    float3 c = centre_of(cdev, chost);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        key[i] = (uint64_t)__float_as_uint(dist2_f32(x[i], y[i], z[i], c.x, c.y, c.z));
}

__global__ void sel_knn_write_k(const int *sorted_idx, int64_t n, int k, const unsigned *gave_up, int *idx, int *count,
                                DevState *st) {
    int kk = *gave_up ? 0 : (int)min((int64_t)k, n);   // the sort gave up: nothing is selected
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < kk; p += gridDim.x * blockDim.x) idx[p] = sorted_idx[p];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *count = kk;
        st->n_pert = kk;
    }
}

// ---------------------------------------------------------------------------
// k nearest by selection: the stars in order of (FP32 squared distance bits,
// caller index), the first k of them, without sorting the rest. (1) counts of the
// distances' leading 11 bits (exponent and three mantissa bits: an eighth of
// an octave a bin); (2) the stars up to the bin that holds the k-th are gathered,
// in any order -- about 1.1 to 1.2 k of them unless many stars lie at nearly
// one distance; (3) one block a member sorts them. If they do not fit its shared
// memory (a centre far outside a compact system sees every star in one bin) the
// blocks of its cluster first narrow them (near_narrow).
// Two reads of the positions instead of a four-pass radix sort of all stars:
// 256 of 2^20 stars 111 -> 30 us of kernels (cold). Members side by side (grid y): a member's
// candidates go to its own slots of the buffer.
// ---------------------------------------------------------------------------
constexpr int kSelCap = 8192;        // candidates a block sorts in shared memory
constexpr int kSelMaxK = kMaxPert;   // larger selections sort everything

struct SelNear {
    const int64_t *moff;      // member offsets (nullptr: one member of n stars)
    int64_t n;
    const float *x, *y, *z;
    const float *cdev;        // centres (x, y, z, .), member m's at 4 (m C + j); nullptr: chost
    int C, j;
    float3 chost;
    int k, cap;               // wanted; slots of a member's output
    int *hist;                // [members][kSelBins]: zero before and after
    int4 *found;              // [members]: candidates, then the bits set and the bits not set in any key
                              // of the k-th's bin; zero before and after
    uint64_t *cand, *alt;     // [n] each
    int *idx, *count;         // chain ch's output at idx + ch cap, count + ch (ch = m C + j)
    DevState *st;
    bool report;              // one member: st->n_pert as well
};

__device__ __forceinline__ int near_bin(unsigned key) { return (int)min(key >> 20, (unsigned)kSelBins - 1); }

__device__ __forceinline__ float3 near_centre(const SelNear &A, int m) {
    const float *q = A.cdev ? A.cdev + 4 * ((int64_t)m * A.C + A.j) : nullptr;
    return q ? make_float3(q[0], q[1], q[2]) : A.chost;
}

// Calls take(key[4], i[4]) for the block's stars, four of a thread's loaded at once,
// whole warps together (i < 0: none).
template <typename F>
__device__ __forceinline__ void near_scan(const SelNear &A, const float3 &c, int64_t s, int64_t e, F &&take) {
    const int64_t stride = (int64_t)gridDim.x * 256;
    for (int64_t b = s + (int64_t)blockIdx.x * 256 + (threadIdx.x & ~31); b < e; b += 4 * stride) {
        unsigned key[4];
        int i[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int64_t q = b + u * stride + (threadIdx.x & 31), j = min(q, e - 1);
            i[u] = q < e ? (int)q : -1;
            key[u] = __float_as_uint(dist2_f32(A.x[j], A.y[j], A.z[j], c.x, c.y, c.z));
        }
        take(key, i);
    }
}

__global__ void __launch_bounds__(256) near_hist_k(SelNear A) {
    __shared__ int h[kSelBins];
    const int m = blockIdx.y;
    for (int b = threadIdx.x; b < kSelBins; b += 256) h[b] = 0;
    const int64_t s = A.moff ? A.moff[m] : 0, e = A.moff ? A.moff[m + 1] : A.n;
    const float3 c = near_centre(A, m);
    __syncthreads();
    near_scan(A, c, s, e, [&](const unsigned *key, const int *i) {
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (i[u] >= 0) atomicAdd(&h[near_bin(key[u])], 1);
    });
    __syncthreads();
    for (int b = threadIdx.x; b < kSelBins; b += 256)
        if (h[b]) atomicAdd(&A.hist[(int64_t)m * kSelBins + b], h[b]);
}

// Inclusive sum over the block of one value a thread (NT threads).
template <int NT>
__device__ __forceinline__ int block_inclusive_sum(int v, int *sw) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sw[wid] = x;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < wid; w++) before += sw[w];
    return before + x;
}

// The first bin at which the running count of h reaches `need` (need >= 1, not
// above the total), and the count before it; the same in every thread.
template <int NT>
__device__ __forceinline__ void find_bin(const int *h, int need, int *sw, int *found, int &bin, int &before) {
    constexpr int PER = kSelBins / NT;
    int v[PER], s = 0;
#pragma unroll
    for (int q = 0; q < PER; q++) {
        v[q] = h[threadIdx.x * PER + q];
        s += v[q];
    }
    const int incl = block_inclusive_sum<NT>(s, sw);
    int run = incl - s;
    if (run < need && incl >= need) {
#pragma unroll
        for (int q = 0; q < PER; q++) {
            if (run < need && run + v[q] >= need) {
                found[0] = threadIdx.x * PER + q;
                found[1] = run;
            }
            run += v[q];
        }
    }
    __syncthreads();
    bin = found[0];
    before = found[1];
}

__global__ void __launch_bounds__(256) near_gather_k(SelNear A) {
    __shared__ int sw[8], found[2];
    const int m = blockIdx.y;
    const int64_t s = A.moff ? A.moff[m] : 0, e = A.moff ? A.moff[m + 1] : A.n;
    const int need = (int)min((int64_t)A.k, e - s);
    if (need <= 0) return;
    int bin, before;
    find_bin<256>(A.hist + (int64_t)m * kSelBins, need, sw, found, bin, before);
    const float3 c = near_centre(A, m);
    unsigned ones = 0, zeros = 0;
    near_scan(A, c, s, e, [&](const unsigned *key, const int *i) {
        bool mine[4], any = false;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            mine[u] = i[u] >= 0 && near_bin(key[u]) <= bin;
            any |= mine[u];
        }
        if (!__any_sync(0xffffffffu, any)) return;
        unsigned in[4];
        int all = 0;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            in[u] = __ballot_sync(0xffffffffu, mine[u]);
            all += __popc(in[u]);
        }
        int at = 0;   // (one place in the list for a warp's four rounds: many candidates queue at one counter)
        if ((threadIdx.x & 31) == 0) at = atomicAdd(&A.found[m].x, all);
        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (mine[u]) {
                A.cand[s + at + __popc(in[u] & lanemask_lt())] = ((uint64_t)key[u] << 32) | (unsigned)i[u];
                if (near_bin(key[u]) == bin) {
                    ones |= key[u];
                    zeros |= ~key[u];
                }
            }
            at += __popc(in[u]);
        }
    });
    ones = __reduce_or_sync(0xffffffffu, ones);
    zeros = __reduce_or_sync(0xffffffffu, zeros);
    if ((threadIdx.x & 31) == 0 && (ones | zeros)) {
        atomicOr(reinterpret_cast<unsigned *>(&A.found[m].y), ones);
        atomicOr(reinterpret_cast<unsigned *>(&A.found[m].z), zeros);
    }
}

// Calls take(ok, value) for this block's share of a candidate list, 32 or 64 KB of it
// loaded at once (a block's reads are bound by their latency), whole warps together.
template <int NT, typename F>
__device__ __forceinline__ void near_share(const uint64_t *a, int rem, int rank, int CL, F &&take) {
    constexpr int U = NT <= 256 ? 16 : 8;
    const int lane = threadIdx.x & 31, stride = NT * CL;
    for (int b = rank * NT + (threadIdx.x & ~31); b < rem; b += U * stride) {
        unsigned long long w[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (b + u * stride + lane < rem)   // (the list of a later round was written by other blocks: from L2)
                w[u] = __ldcg(reinterpret_cast<const unsigned long long *>(a) + b + u * stride + lane);
#pragma unroll
        for (int u = 0; u < U; u++) take(b + u * stride + lane < rem, (uint64_t)w[u]);
    }
}

struct NearSmem {
    int h[kSelBins], sw[32], found[2], nacc, nrem;
};

// Narrows `rem` candidates (list a) to what a block sorts, digit by digit of the
// 64-bit (distance, index) value, which is different for every star, so this
// ends for any input: what lies below the digit of the k-th goes to the first
// block's array v (fewer than `want` in all), what shares it to the other list.
// The CL blocks of a member's cluster share the lists; the counts and v are the
// first block's. On return v holds acc values and list a the other rem. shift: the
// first digit's.
template <int NT>
__device__ void near_narrow(NearSmem &S, int shift, uint64_t *v, uint64_t *&a, uint64_t *o, int want, int rank,
                            int CL, int &acc, int &rem) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x;
    int *h0 = cl.map_shared_rank(S.h, 0), *nacc0 = cl.map_shared_rank(&S.nacc, 0),
        *nrem0 = cl.map_shared_rank(&S.nrem, 0);
    uint64_t *v0 = cl.map_shared_rank(v, 0);
    // the next places of the set lanes at a counter of the first block
    auto slots = [](int *counter, unsigned set) -> int {
        int at = 0;
        if ((threadIdx.x & 31) == 0) at = atomicAdd(counter, __popc(set));
        return __shfl_sync(0xffffffffu, at, 0) + __popc(set & lanemask_lt());
    };
    if (t == 0) S.nacc = 0;
    for (; acc + rem > kSelCap; shift = max(shift - 11, 0)) {
        auto digit = [&](uint64_t w) -> int { return (int)(w >> shift) & (kSelBins - 1); };
        for (int b = t; b < kSelBins; b += NT) S.h[b] = 0;
        cl.sync();
        if (t == 0) S.nrem = 0;
        near_share<NT>(a, rem, rank, CL, [&](bool ok, uint64_t w) {
            if (ok) atomicAdd(&S.h[digit(w)], 1);
        });
        __syncthreads();
        if (rank != 0)
            for (int b = t; b < kSelBins; b += NT)
                if (S.h[b]) atomicAdd(h0 + b, S.h[b]);
        cl.sync();
        if (rank != 0)
            for (int b = t; b < kSelBins; b += NT) S.h[b] = h0[b];
        __syncthreads();
        int bin, before;
        find_bin<NT>(S.h, want - acc, S.sw, S.found, bin, before);
        if (S.h[bin] != rem) {   // (all share the digit: nothing to move)
            near_share<NT>(a, rem, rank, CL, [&](bool ok, uint64_t w) {
                const int d = ok ? digit(w) : kSelBins;
                const unsigned below = __ballot_sync(0xffffffffu, d < bin), same = __ballot_sync(0xffffffffu, d == bin);
                if (below) {
                    const int at = slots(nacc0, below);
                    if (d < bin) v0[at] = w;
                }
                if (same) {
                    const int at = slots(nrem0, same);
                    if (d == bin) o[at] = w;
                }
            });
            cl.sync();
            acc = *nacc0;
            rem = *nrem0;
            uint64_t *q = a;
            a = o;
            o = q;
        }
        cl.sync();   // the first block's counts are read before it goes on
    }
}

// Grid: CL blocks a member (a cluster); the first one sorts, the others only
// help to narrow.
template <int NT>
__global__ void __launch_bounds__(NT) near_sort_k(SelNear A, int CL) {
    extern __shared__ __align__(16) char near_smem[];
    uint64_t *v = reinterpret_cast<uint64_t *>(near_smem);   // [kSelCap]
    __shared__ NearSmem S;
    const int m = blockIdx.x / CL, rank = blockIdx.x % CL, t = threadIdx.x;
    const int64_t s = A.moff ? A.moff[m] : 0, e = A.moff ? A.moff[m + 1] : A.n;
    const int64_t ch = (int64_t)m * A.C + A.j;
    int *hist = A.hist + (int64_t)m * kSelBins;
    const int take = (int)min((int64_t)A.k, e - s);
    // (few candidates: the first block may clear the count before the others read it, and
    // they end either way; many: it is cleared after the cluster has met)
    int rem = take > 0 ? *(volatile int *)&A.found[m].x : 0, acc = 0;
    if (rank != 0 && rem <= kSelCap) return;
    __syncthreads();
    uint64_t *a = A.cand + s;
    if (rem > kSelCap) {
        // all candidates in the k-th's bin: they share its bits (the last bin holds several values),
        // and the first digit starts at the highest bit in which any two differ
        int bin, before, shift = 53;
        find_bin<NT>(hist, take, S.sw, S.found, bin, before);
        if (before == 0 && bin < kSelBins - 1) {
            const unsigned differ = (unsigned)A.found[m].y & (unsigned)A.found[m].z;
            const int top = differ ? 63 - __clz(differ) : 31 - __clz((int)(e - 1));
            shift = max(top - 10, 0);
        }
        near_narrow<NT>(S, shift, v, a, A.alt + s, take, rank, CL, acc, rem);
    }
    if (rank != 0) return;
    for (int b = t; b < kSelBins; b += NT) hist[b] = 0;   // ready for the next selection
    if (t == 0) A.found[m] = make_int4(0, 0, 0, 0);
    for (int i = t; i < rem; i += NT) v[acc + i] = __ldcg(reinterpret_cast<const unsigned long long *>(a) + i);
    int size = 2;
    while (size < acc + rem) size <<= 1;
    for (int i = acc + rem + t; i < size; i += NT) v[i] = ~0ull;
    __syncthreads();
    // bitonic sort; pairs up to 32 apart stay within a warp's 64 elements, so only
    // longer strides, and the step from one back to them, need the block's barrier
    for (int k = 2; k <= size; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int q = t; q < size / 2; q += NT) {
                const int i = 2 * q - (q & (j - 1));   // the pair's lower place
                const uint64_t lo = v[i], hi = v[i + j];
                if ((lo > hi) == ((i & k) == 0)) {
                    v[i] = hi;
                    v[i + j] = lo;
                }
            }
            if (j > 32 || (j == 1 && k >= 64)) __syncthreads();
            else __syncwarp();
        }
    __syncthreads();
    const int kk = min(take, A.cap);
    for (int i = t; i < kk; i += NT) A.idx[ch * A.cap + i] = (int)(unsigned)v[i];
    if (t == 0) {
        A.count[ch] = kk;
        if (A.report) A.st->n_pert = kk;
        else if (take > A.cap) latch_err(A.st, kErrPert);
    }
}

// Blocks of a cluster that narrow a member's candidates together: one block reads
// them at the rate of its latency (25 GB/s). us a search of 256, 4000 of 2^20 stars
// from 1000 and 10^6 radii away, one block | eight | a sort of all stars: 57, 740
// and 2280, 720 | 60, 124 and 126, 106 | 156 and 144. From inside the system, where a block's
// memory holds the candidates, nothing changes (27 us; the other blocks end at
// once). A block alone does for systems of up to 2^14 stars (from outside 85 to 95 us
// of 5000), and in an ensemble, whose blocks are many, for members of up to 2^16.
constexpr int kSelBlocks = 8;
static int near_blocks(int members, int64_t largest, int sms) {
    return largest > (members == 1 ? 1 << 14 : 1 << 16) && members * kSelBlocks <= 2 * sms ? kSelBlocks : 1;
}

template <int NT>
static cudaError_t near_sort(const SelNear &A, int members, int CL, cudaStream_t s) {
    const size_t smem = sizeof(uint64_t) * kSelCap;
    cudaError_t e = cudaFuncSetAttribute(near_sort_k<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(members * CL);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, near_sort_k<NT>, A, CL);
}

static rv_status select_nearest(rv_ctx *c, const SelNear &A, int members, int64_t largest, cudaStream_t s) {
    // (few candidates: a small block, whose barriers are cheaper)
    const bool few = std::min(A.k, A.cap) <= 512;
    const int CL = near_blocks(members, largest, c->num_sms);
    // about 1024 stars a block, four blocks an SM over all members
    const int bx = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(largest, 1024), (int64_t)c->num_sms * 4 / members + 1));
    near_hist_k<<<dim3(bx, members), 256, 0, s>>>(A);
    near_gather_k<<<dim3(bx, members), 256, 0, s>>>(A);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = few ? near_sort<256>(A, members, CL, s) : near_sort<1024>(A, members, CL, s);
    c->launches += 3;
    return cuda_check(c, e, "select nearest");
}

// Eq. 1 ingredients from the stars sorted by FP32 squared distance (keys =
// the d2 bits, ties by index): r(<2 M_bh), sigma of the k nearest, M_bh / sigma^2.
// One thread, sums in distance order in FP64, exactly as the rule reads. out[3] =
// 1 if the sort gave up (nothing else is written then).
__global__ void influence_k(int64_t n, const uint64_t *skey, const int *sidx, const float *vx, const float *vy,
                            const float *vz, const float *m, double m_bh, int64_t k, const unsigned *gave_up,
                            double *out) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    out[3] = *gave_up ? 1.0 : 0.0;
    if (*gave_up) return;
    double cum = 0.0, r2m = __longlong_as_double(0x7ff0000000000000ll);
    for (int64_t i = 0; i < n; i++) {
        cum = __dadd_rn(cum, (double)m[sidx[i]]);
        if (cum >= 2.0 * m_bh) {
            r2m = __dsqrt_rn((double)__uint_as_float((unsigned)skey[i]));
            break;
        }
    }
    double mx = 0.0, my = 0.0, mz = 0.0;
    for (int64_t i = 0; i < k; i++) {
        const int j = sidx[i];
        mx = __dadd_rn(mx, (double)vx[j]); my = __dadd_rn(my, (double)vy[j]); mz = __dadd_rn(mz, (double)vz[j]);
    }
    mx = __ddiv_rn(mx, (double)k); my = __ddiv_rn(my, (double)k); mz = __ddiv_rn(mz, (double)k);
    double s = 0.0;
    for (int64_t i = 0; i < k; i++) {
        const int j = sidx[i];
        const double dx = __dsub_rn((double)vx[j], mx), dy = __dsub_rn((double)vy[j], my),
                     dz = __dsub_rn((double)vz[j], mz);
        s = __dadd_rn(s, __dmul_rn(dx, dx));
        s = __dadd_rn(s, __dmul_rn(dy, dy));
        s = __dadd_rn(s, __dmul_rn(dz, dz));
    }
    const double s2 = __ddiv_rn(s, __dmul_rn(3.0, (double)k));
    out[0] = r2m;
    out[1] = __dsqrt_rn(s2);
    out[2] = __ddiv_rn(m_bh, s2);
}

static int grid_n(rv_ctx *c, int64_t n) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)c->num_sms * 8));
}

rv_status select_perturbers(rv_ctx *c, int64_t n, const float *x, const float *y, const float *z,
                            const float *centre_dev, const float *centre_host, int mode, float radius, int k,
                            int cap, int *idx, int *count, cudaStream_t s, const float *m, float gamma) {
    // centre_host: (x, y, z, chain mass) -- the mass is read by the tidal rule only
    float4 ch = centre_host ? make_float4(centre_host[0], centre_host[1], centre_host[2], centre_host[3])
                            : make_float4(0, 0, 0, 0);
    Workspace &w = c->w;
    if (mode == 1 || mode == 3) {
        const SelRule R = sel_rule(mode, radius, m, gamma);
        if (n == 0) return cuda_check(c, cudaMemsetAsync(count, 0, sizeof(int), s), "select");
        int *total = &w.st->n_pert;
        sel_radius_flag_k<<<grid_n(c, n), 256, 0, s>>>(n, x, y, z, centre_dev, ch, R, w.sel_flag, total);
        count_launch(c);
        rv_status r = exclusive_scan(c, w.sel_flag, n, total, s);
        if (r != RV_OK) return r;
        sel_radius_write_k<<<grid_n(c, n), 256, 0, s>>>(n, x, y, z, centre_dev, ch, R, w.sel_flag, total, cap, idx,
                                                        count, w.st);
        count_launch(c);
    } else {
        if (n == 0 || k <= 0) {
            cudaMemsetAsync(&w.st->n_pert, 0, sizeof(int), s);
            return cuda_check(c, cudaMemsetAsync(count, 0, sizeof(int), s), "select");
        }
        // the sort buffers are shared with the tree build: the tree is invalid afterwards
        c->built = false;
        if (std::min<int64_t>(k, n) <= kSelMaxK) {
            // (one member: an output shorter than k is simply the nearest cap of them)
            const SelNear A{nullptr, n, x, y, z, centre_dev, 1, 0, make_float3(ch.x, ch.y, ch.z), std::min(k, cap), cap,
                            w.selhist, w.selfound, w.key_a, w.key_b, idx, count, w.st, true};
            if (A.k > 0) return select_nearest(c, A, 1, n, s);
        }
        sel_knn_keys_k<<<grid_n(c, n), 256, 0, s>>>(n, x, y, z, centre_dev, make_float3(ch.x, ch.y, ch.z), w.key_a);
        count_launch(c);
        uint64_t *sk;
        int *si;
        rv_status r = radix_sort(c, n, 4, &sk, &si, s);
        if (r != RV_OK) return r;
        sel_knn_write_k<<<ceil_div(std::min<int64_t>(k, n), 256), 256, 0, s>>>(si, n, std::min(k, cap), w.lb + kLbGaveUp,
                                                                                      idx, count, w.st);
        count_launch(c);
    }
    return cuda_check(c, cudaGetLastError(), "select perturbers");
}

rv_status influence_radius(rv_ctx *c, int64_t n, const float *x, const float *y, const float *z, const float *vx,
                           const float *vy, const float *vz, const float *m, const float centre[3], double m_bh,
                           int64_t n_sigma, double out[3], cudaStream_t s) {
    Workspace &w = c->w;
    c->built = false;   // the sort buffers are shared with the tree build
    sel_knn_keys_k<<<grid_n(c, n), 256, 0, s>>>(n, x, y, z, nullptr, make_float3(centre[0], centre[1], centre[2]),
                                                w.key_a);
    count_launch(c);
    uint64_t *sk;
    int *si;
    rv_status r = radix_sort(c, n, 4, &sk, &si, s);
    if (r != RV_OK) return r;
    influence_k<<<1, 32, 0, s>>>(n, sk, si, vx, vy, vz, m, m_bh, std::min<int64_t>(n_sigma, n),
                                 w.lb + kLbGaveUp, w.out8);
    count_launch(c);
    double res[4] = {0, 0, 0, 0};
    r = cuda_check(c, cudaMemcpyAsync(res, w.out8, sizeof res, cudaMemcpyDeviceToHost, s), "influence");
    if (r == RV_OK) r = cuda_check(c, cudaStreamSynchronize(s), "influence");
    if (r != RV_OK) return r;
    if (res[3] != 0.0) return set_err(c, RV_E_TIMEOUT, "a wait of the star sort gave up");
    for (int k = 0; k < 3; k++) out[k] = res[k];
    return RV_OK;
}

// ---------------------------------------------------------------------------
// radius or tidal search per member (systems of several members): one stable
// sort of (member, key) over all stars, key = 0 inside, 1 outside; member m's stars
// occupy the same slots [moff[m], moff[m+1]) in sorted order, inside ones first
// in ascending index.
// ---------------------------------------------------------------------------
__global__ void sel_member_keys_k(const int64_t *moff, int bpm, const float *x, const float *y, const float *z,
                                  const float *xyzm, int C, int j, SelRule R, uint64_t *key) {
    const int m = blockIdx.y;
    const float *q = xyzm + 4 * ((int64_t)m * C + j);   // chain j of member m
    const float cx = q[0], cy = q[1], cz = q[2], mc = q[3];
    for (int64_t i = moff[m] + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < moff[m + 1];
         i += (int64_t)bpm * blockDim.x) {
        float d2 = dist2_f32(x[i], y[i], z[i], cx, cy, cz);
        key[i] = sel_inside(R, d2, i, mc) ? 0ull : 1ull;
    }
}

// member m: its leading "inside" slots, written to idx[m cap ..], count to npert[m]
__global__ void sel_member_write_k(const int64_t *moff, const uint64_t *skey, const int *sidx, int cap, int C, int j, const unsigned *gave_up, int *idx, int *npert, DevState *st) {
    const int m = blockIdx.x;
    const int64_t s = moff[m], e = moff[m + 1];
    int cnt = 0;
    if (!*gave_up) {   // (a sort that gave up: nothing is selected)
        // first "outside" key in the member's slots
        int64_t lo = s, hi = e;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if (skey[mid] == 0ull) lo = mid + 1; else hi = mid;
        }
        cnt = (int)(lo - s);
    }
    if (cnt > cap && threadIdx.x == 0) latch_err(st, kErrPert);
    cnt = min(cnt, cap);
    const int64_t ch = (int64_t)m * C + j;   // chain j of member m
    for (int p = threadIdx.x; p < cnt; p += blockDim.x) idx[ch * cap + p] = sidx[s + p];
    if (threadIdx.x == 0) npert[ch] = cnt;
}

static int member_cap(int M) { return std::min(kMaxPert, kPertTotal / std::max(1, M)); }

// ---------------------------------------------------------------------------
// FP64 chain / perturber coupling, one chain per member
// ---------------------------------------------------------------------------
// f = m r / |r|^3 and -m/|r| for r = to - from (zero separation: nothing).
__device__ __forceinline__ void kep(double rx, double ry, double rz, double m, double &ax, double &ay, double &az,
                                    double &p) {
    double r2 = rx * rx + ry * ry + rz * rz;
    if (r2 <= 0.0) return;
    double rinv = 1.0 / sqrt(r2);
    double s = m * rinv * rinv * rinv;
    ax += s * rx; ay += s * ry; az += s * rz;
    p -= m * rinv;
}

// Per member m (out8 + 16 m): [0..3) corr (Eq. 3), [3..6) sub, [6] sum_k m_k
// pot_chain[k] / M, [7] sub potential, [8..11) centre of mass, [11] M.
// With xyzm, the centre of mass also becomes member m's extra particle m
// (FP32, unsoftened). With xq, the chain's traceless quadrupole about its
// centre of mass, Q_ab = sum_k m_k (3 d_a d_b - |d|^2 delta_ab), d = x_k - c
// (the expansion of Sect. 1 applied to the chain), computed in FP64, goes
// rounded to FP32 to xq[2 m] = (xx, yy, zz, xy), xq[2 m + 1] = (xz, yz, 0, 0)
// for the walk.
__global__ void chain_com_k(int M, int n_ch, const double *cm, const double *cx, double *out8, float *xyzm,
                            float *xeps, float4 *xq = nullptr) {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) {
        const double *mm = cm + (int64_t)m * n_ch, *xx = cx + 3 * (int64_t)m * n_ch;
        double Mt = 0, c[3] = {0, 0, 0};
        for (int k = 0; k < n_ch; k++) {
            Mt += mm[k];
            for (int a = 0; a < 3; a++) c[a] += mm[k] * xx[3 * k + a];
        }
        for (int a = 0; a < 3; a++) c[a] = (Mt > 0) ? c[a] / Mt : 0.0;
        double *o = out8 + 16 * (int64_t)m;
        o[8] = c[0]; o[9] = c[1]; o[10] = c[2]; o[11] = Mt;
        if (xyzm) {
            xyzm[4 * m] = (float)c[0]; xyzm[4 * m + 1] = (float)c[1]; xyzm[4 * m + 2] = (float)c[2];
            xyzm[4 * m + 3] = (float)Mt;
            xeps[m] = 0.f;
        }
        if (xq) {
            double q[6] = {0, 0, 0, 0, 0, 0};
            for (int k = 0; k < n_ch; k++) {
                const double d0 = xx[3 * k] - c[0], d1 = xx[3 * k + 1] - c[1], d2 = xx[3 * k + 2] - c[2];
                const double dd = d0 * d0 + d1 * d1 + d2 * d2;
                q[0] += mm[k] * (3.0 * d0 * d0 - dd);
                q[1] += mm[k] * (3.0 * d1 * d1 - dd);
                q[2] += mm[k] * (3.0 * d2 * d2 - dd);
                q[3] += mm[k] * 3.0 * d0 * d1;
                q[4] += mm[k] * 3.0 * d0 * d2;
                q[5] += mm[k] * 3.0 * d1 * d2;
            }
            xq[2 * m] = make_float4((float)q[0], (float)q[1], (float)q[2], (float)q[3]);
            xq[2 * m + 1] = make_float4((float)q[4], (float)q[5], 0.f, 0.f);
        }
    }
}

// Member addressing shared by the coupling kernels (blockIdx.y = member).
struct ChainView {
    int n_ch;            // members of each chain
    int cap;             // perturber slots per member
    const double *cm, *cx;
    const int *npert;    // perturbers per member (nullptr: cap)
    const double *pm, *px;
};

__device__ __forceinline__ int npert_of(const ChainView &V, int m) { return V.npert ? min(V.npert[m], V.cap) : V.cap; }

// perturbers: resolved members minus the centre-of-mass point mass (the walk
// gives perturbers the point mass only, never the chain's quadrupole)
__global__ void pert_on_stars_k(ChainView V, const double *out8, double *a_pert, double *pot_pert) {
    const int m = blockIdx.y;
    const int np = npert_of(V, m);
    const double *cm = V.cm + (int64_t)m * V.n_ch, *cx = V.cx + 3 * (int64_t)m * V.n_ch;
    const double *o = out8 + 16 * (int64_t)m;
    const double M = o[11];
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const int64_t q = (int64_t)m * V.cap + p;
        double x = V.px[3 * q], y = V.px[3 * q + 1], z = V.px[3 * q + 2];
        double ax = 0, ay = 0, az = 0, ph = 0;
        for (int k = 0; k < V.n_ch; k++) kep(cx[3 * k] - x, cx[3 * k + 1] - y, cx[3 * k + 2] - z, cm[k], ax, ay, az, ph);
        double bx = 0, by = 0, bz = 0, bp = 0;
        kep(o[8] - x, o[9] - y, o[10] - z, M, bx, by, bz, bp);
        a_pert[3 * q] = ax - bx; a_pert[3 * q + 1] = ay - by; a_pert[3 * q + 2] = az - bz;
        pot_pert[q] = ph - bp;
    }
}

template <int NT>
__device__ void block_sum4(double v[4], double (*sm)[NT]) {
    for (int a = 0; a < 4; a++) sm[a][threadIdx.x] = v[a];
    __syncthreads();
    for (int o = NT / 2; o >= 32; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int a = 0; a < 4; a++) sm[a][threadIdx.x] += sm[a][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 32) {   // the last five halvings within a warp
        for (int a = 0; a < 4; a++) {
            double s = sm[a][threadIdx.x];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (threadIdx.x == 0) sm[a][0] = s;
        }
    }
    __syncthreads();
    for (int a = 0; a < 4; a++) v[a] = sm[a][0];
    __syncthreads();
}

// block (k, m): perturbers of member m on its chain member k (fixed order)
__global__ void __launch_bounds__(256) pert_on_members_k(ChainView V, double *a_chain, double *pot_chain) {
    __shared__ double sm[4][256];
    const int k = blockIdx.x, m = blockIdx.y;
    const int np = npert_of(V, m);
    const int64_t kk = (int64_t)m * V.n_ch + k;
    double x = V.cx[3 * kk], y = V.cx[3 * kk + 1], z = V.cx[3 * kk + 2];
    double v[4] = {0, 0, 0, 0};
    for (int p = threadIdx.x; p < np; p += 256) {
        const int64_t q = (int64_t)m * V.cap + p;
        kep(V.px[3 * q] - x, V.px[3 * q + 1] - y, V.px[3 * q + 2] - z, V.pm[q], v[0], v[1], v[2], v[3]);
    }
    block_sum4<256>(v, sm);
    if (threadIdx.x == 0) {
        a_chain[3 * kk] = v[0]; a_chain[3 * kk + 1] = v[1]; a_chain[3 * kk + 2] = v[2];
        pot_chain[kk] = v[3];
    }
}

// block m: Eq. 3 correction, and the perturbers' direct terms on the centre of mass
__global__ void __launch_bounds__(256) pert_totals_k(ChainView V, const double *a_chain, const double *pot_chain,
                                                     double *out8) {
    __shared__ double sm[4][256];
    const int m = blockIdx.x;
    const int np = npert_of(V, m);
    double *o = out8 + 16 * (int64_t)m;
    const double M = o[11];
    double v[4] = {0, 0, 0, 0};
    for (int k = threadIdx.x; k < V.n_ch; k += 256) {
        const int64_t kk = (int64_t)m * V.n_ch + k;
        const double mk = V.cm[kk];
        v[0] += mk * a_chain[3 * kk]; v[1] += mk * a_chain[3 * kk + 1]; v[2] += mk * a_chain[3 * kk + 2];
        v[3] += mk * pot_chain[kk];
    }
    block_sum4<256>(v, sm);
    double u[4] = {0, 0, 0, 0};
    for (int p = threadIdx.x; p < np; p += 256) {
        const int64_t q = (int64_t)m * V.cap + p;
        kep(V.px[3 * q] - o[8], V.px[3 * q + 1] - o[9], V.px[3 * q + 2] - o[10], V.pm[q], u[0], u[1], u[2], u[3]);
    }
    block_sum4<256>(u, sm);
    if (threadIdx.x == 0) {
        for (int a = 0; a < 3; a++) o[a] = (M > 0) ? v[a] / M : 0.0;
        for (int a = 0; a < 3; a++) o[3 + a] = u[a];
        o[6] = (M > 0) ? v[3] / M : 0.0;
        o[7] = u[3];
    }
}

static rv_status coupling(rv_ctx *c, int M, const ChainView &V, double *a_pert, double *pot_pert, double *a_chain,
                          double *pot_chain, double *out8, cudaStream_t s) {
    chain_com_k<<<ceil_div(M, 128), 128, 0, s>>>(M, V.n_ch, V.cm, V.cx, out8, nullptr, nullptr);
    count_launch(c);
    if (V.cap > 0) {
        pert_on_stars_k<<<dim3(ceil_div(V.cap, 128), M), 128, 0, s>>>(V, out8, a_pert, pot_pert);
        count_launch(c);
    }
    if (V.n_ch > 0) {
        pert_on_members_k<<<dim3(V.n_ch, M), 256, 0, s>>>(V, a_chain, pot_chain);
        count_launch(c);
    }
    pert_totals_k<<<M, 256, 0, s>>>(V, a_chain, pot_chain, out8);
    count_launch(c);
    return cuda_check(c, cudaGetLastError(), "perturber forces");
}

rv_status perturber_forces(rv_ctx *c, int n_ch, const double *cm, const double *cx, int n_pert_max,
                           const int *d_npert, const double *pm, const double *px, double *a_pert,
                           double *pot_pert, double *a_chain, double *pot_chain, double *out8, cudaStream_t s) {
    ChainView V{n_ch, n_pert_max, cm, cx, d_npert, pm, px};
    return coupling(c, 1, V, a_pert, pot_pert, a_chain, pot_chain, out8, s);
}

// ---------------------------------------------------------------------------
// system force evaluation
// ---------------------------------------------------------------------------
__global__ void gather_pert_k(int cap, const int *idx, const int *npert, const float *x, const float *y,
                              const float *z, const float *m, double *pm, double *px) {
    const int mb = blockIdx.y;
    const int np = min(npert[mb], cap);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const int64_t q = (int64_t)mb * cap + p;
        const int i = idx[q];
        pm[q] = (double)m[i];
        px[3 * q] = (double)x[i]; px[3 * q + 1] = (double)y[i]; px[3 * q + 2] = (double)z[i];
    }
}

// flag[i] = 1 for every star that is a perturber of some chain (the walk gives
// those no chain quadrupole: they feel the resolved members instead)
__global__ void mark_pert_k(int cap, const int *idx, const int *npert, uint8_t *flag) {
    const int mb = blockIdx.y;
    const int np = min(npert[mb], cap);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x)
        flag[idx[(int64_t)mb * cap + p]] = 1;
}

// perturbers of the last selection predicted to first order, dt after the force pass
// (Sect. 2: the chain integrator predicts them at each of its force evaluations):
// x_p(dt) = x_p + v_p dt in FP64, one rounding per operation
__global__ void predict_pert_k(int cap, const int *idx, const int *npert, const float *x, const float *y,
                               const float *z, const float *vx, const float *vy, const float *vz, const float *m,
                               double dt, double *pm, double *px) {
    const int mb = blockIdx.y;
    const int np = min(npert[mb], cap);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const int64_t q = (int64_t)mb * cap + p;
        const int i = idx[q];
        pm[q] = (double)m[i];
        px[3 * q] = __dadd_rn((double)x[i], __dmul_rn((double)vx[i], dt));
        px[3 * q + 1] = __dadd_rn((double)y[i], __dmul_rn((double)vy[i], dt));
        px[3 * q + 2] = __dadd_rn((double)z[i], __dmul_rn((double)vz[i], dt));
    }
}

// stars that are perturbers: add the FP64 correction (resolved chain - centre-of-mass point mass)
// (block time steps: only the stars active now, whose forces this pass wrote)
__global__ void apply_pert_k(int cap, const int *idx, const int *npert, const double *a_pert, const double *pot_pert,
                             float *ax, float *ay, float *az, float *pot, const int8_t *level, long long n, int L) {
    const int mb = blockIdx.y;
    const int np = min(npert[mb], cap);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const int64_t q = (int64_t)mb * cap + p;
        const int i = idx[q];
        if (level && (n & ((1ll << (L - min(max((int)level[i], 0), L))) - 1)) != 0) continue;
        ax[i] = (float)((double)ax[i] + a_pert[3 * q]);
        ay[i] = (float)((double)ay[i] + a_pert[3 * q + 1]);
        az[i] = (float)((double)az[i] + a_pert[3 * q + 2]);
        pot[i] = (float)((double)pot[i] + pot_pert[q]);
    }
}

// Chain member k of member m: mutual unsoftened FP64 pull of the other chain
// members, plus the perturbers on k, plus the tree's force on the centre of
// mass without the perturbers' direct terms (those are resolved per member).
__global__ void chain_accel_k(int M, int n_ch, const double *cm, const double *cx, const double *a_ext,
                              const double *pot_ext, const float *xout, const double *out8, double *ca, double *cpot) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < M * n_ch; t += gridDim.x * blockDim.x) {
        const int m = t / n_ch, k = t % n_ch;
        const double *o = out8 + 16 * (int64_t)m;
        const double *mm = cm + (int64_t)m * n_ch, *xx = cx + 3 * (int64_t)m * n_ch;
        double tx = (double)xout[4 * m] - o[3], ty = (double)xout[4 * m + 1] - o[4], tz = (double)xout[4 * m + 2] - o[5];
        double tp = (double)xout[4 * m + 3] - o[7];
        double ax = 0, ay = 0, az = 0, ph = 0;
        for (int j = 0; j < n_ch; j++) {
            if (j == k) continue;
            kep(xx[3 * j] - xx[3 * k], xx[3 * j + 1] - xx[3 * k + 1], xx[3 * j + 2] - xx[3 * k + 2], mm[j], ax, ay, az,
                ph);
        }
        ca[3 * (int64_t)t] = ax + a_ext[3 * (int64_t)t] + tx;
        ca[3 * (int64_t)t + 1] = ay + a_ext[3 * (int64_t)t + 1] + ty;
        ca[3 * (int64_t)t + 2] = az + a_ext[3 * (int64_t)t + 2] + tz;
        cpot[t] = ph + pot_ext[t] + tp;
    }
}

// Prediction and pull in one launch, for chains of few members (each block
// predicts the perturbers for itself; the operations are those of predict_pert_k
// and pert_on_members_k). A substep of a pair with 256 perturbers is two short
// kernels otherwise: 12 us a call, 7 in one.
constexpr int kPredictFused = 8;   // members of a chain up to which predicting again costs less than a launch
__global__ void __launch_bounds__(256) predict_on_members_k(int n_ch, int cap, const int *idx, const int *npert,
                                                            const float *x, const float *y, const float *z,
                                                            const float *vx, const float *vy, const float *vz,
                                                            const float *m, double dt, const double *cx, double *a_chain,
                                                            double *pot_chain) {
    __shared__ double sm[4][256];
    const int mb = blockIdx.y;
    const int np = min(npert[mb], cap);
    const int64_t kk = (int64_t)mb * n_ch + blockIdx.x;
    const double px = cx[3 * kk], py = cx[3 * kk + 1], pz = cx[3 * kk + 2];
    double v[4] = {0, 0, 0, 0};
    for (int p = threadIdx.x; p < np; p += 256) {
        const int i = idx[(int64_t)mb * cap + p];
        const double qx = __dadd_rn((double)x[i], __dmul_rn((double)vx[i], dt));
        const double qy = __dadd_rn((double)y[i], __dmul_rn((double)vy[i], dt));
        const double qz = __dadd_rn((double)z[i], __dmul_rn((double)vz[i], dt));
        kep(qx - px, qy - py, qz - pz, (double)m[i], v[0], v[1], v[2], v[3]);
    }
    block_sum4<256>(v, sm);
    if (threadIdx.x == 0) {
        a_chain[3 * kk] = v[0]; a_chain[3 * kk + 1] = v[1]; a_chain[3 * kk + 2] = v[2];
        pot_chain[kk] = v[3];
    }
}

static const int64_t *system_offsets(const rv_system *sys, int64_t tmp[2]);

// Perturber pull on the chain members at chain positions chain_x (member-major
// FP64), the perturbers of the last force pass predicted dt ahead.
rv_status chain_perturber_forces(rv_ctx *c, const rv_system *sys, double dt, const double *chain_x, double *a_chain,
                                 double *pot_chain, cudaStream_t s) {
    Workspace &w = c->w;
    const int M = system_chains(sys);   // the coupling kernels treat each chain as a unit
    const int cap = member_cap(M);
    if (sys->n_chain <= kPredictFused) {
        predict_on_members_k<<<dim3(sys->n_chain, M), 256, 0, s>>>(
            sys->n_chain, cap, w.pert_idx, w.npert, sys->x, sys->y, sys->z, sys->vx, sys->vy, sys->vz, sys->m, dt, chain_x,
            a_chain, pot_chain ? pot_chain : w.chain_ext_pot);
        count_launch(c);
        return cuda_check(c, cudaGetLastError(), "chain perturber forces");
    }
    predict_pert_k<<<dim3(ceil_div(cap, 128), M), 128, 0, s>>>(cap, w.pert_idx, w.npert, sys->x, sys->y, sys->z,
                                                               sys->vx, sys->vy, sys->vz, sys->m, dt, w.pert_m,
                                                               w.pert_x);
    count_launch(c);
    ChainView V{sys->n_chain, cap, sys->chain_m, chain_x, w.npert, w.pert_m, w.pert_x};
    pert_on_members_k<<<dim3(sys->n_chain, M), 256, 0, s>>>(V, a_chain, pot_chain ? pot_chain : w.chain_ext_pot);
    count_launch(c);
    return cuda_check(c, cudaGetLastError(), "chain perturber forces");
}

static const int64_t *system_offsets(const rv_system *sys, int64_t tmp[2]) {
    if (sys->n_members > 1 || sys->member_offsets) return sys->member_offsets;
    tmp[0] = 0;
    tmp[1] = sys->n;
    return tmp;
}

int system_members(const rv_system *sys) { return std::max(1, (int)sys->n_members); }
int chains_per_member(const rv_system *sys) { return std::max(1, (int)sys->n_chains); }
int system_chains(const rv_system *sys) {
    return sys->n_chain > 0 ? system_members(sys) * chains_per_member(sys) : 0;
}

rv_status system_forces(rv_ctx *c, rv_system *sys, cudaStream_t s, const BlockSel *blk) {
    Workspace &w = c->w;
    rv_status r;
    const bool chain = sys->n_chain > 0;
    const int M = system_members(sys);
    const int C = chains_per_member(sys);
    const int NC = system_chains(sys);   // chains: the unit of every chain kernel below
    int64_t tmp[2];
    const int64_t *off = system_offsets(sys, tmp);
    const int cap = member_cap(std::max(1, NC));
    // the chain's quadrupole acts on the stars beyond its perturbers (rv_system.chain_quad)
    const bool quad = chain && sys->chain_quad != 0 && sys->n_chain > 1;
    if (chain) {
        chain_com_k<<<ceil_div(NC, 128), 128, 0, s>>>(NC, sys->n_chain, sys->chain_m, sys->chain_x, w.out8,
                                                      w.extra_xyzm, w.extra_eps, quad ? w.extra_quad : nullptr);
        count_launch(c);
    }
    if ((r = upload_offsets(c, M, off, s)) != RV_OK) return r;
    if (chain && (sys->pert_mode == 1 || sys->pert_mode == 2 || sys->pert_mode == 3)) {
        // one selection per chain j of every member (perturber slots of chain m C + j)
        for (int j = 0; j < C; j++) {
            if (M == 1) {
                r = select_perturbers(c, sys->n, sys->x, sys->y, sys->z, w.extra_xyzm + 4 * j, nullptr,
                                      sys->pert_mode, sys->pert_radius, sys->pert_k, cap, w.pert_idx + (int64_t)j * cap,
                                      w.npert + j, s, sys->m, sys->pert_gamma);
                if (r != RV_OK) return r;
            } else {
                // the sort buffers are shared with the tree build, which comes next
                if (sys->pert_mode == 2) {
                    if (sys->pert_k <= 0) {   // (every chain's count at once)
                        r = cuda_check(c, cudaMemsetAsync(w.npert, 0, sizeof(int) * NC, s), "select nearest");
                        if (r != RV_OK) return r;
                        continue;
                    }
                    const SelNear A{w.moff, sys->n, sys->x, sys->y, sys->z, w.extra_xyzm, C, j, make_float3(0.f, 0.f, 0.f),
                                    sys->pert_k, cap, w.selhist, w.selfound, w.key_a, w.key_b, w.pert_idx, w.npert, w.st,
                                    false};
                    int64_t big = 1;
                    for (int k = 0; k < M; k++) big = std::max<int64_t>(big, off[k + 1] - off[k]);
                    if ((r = select_nearest(c, A, M, big, s)) != RV_OK) return r;
                    continue;
                }
                const int bpm = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(c->max_member, 256), 64));
                const SelRule R = sel_rule(sys->pert_mode, sys->pert_radius, sys->m, sys->pert_gamma);
                sel_member_keys_k<<<dim3(bpm, M), 256, 0, s>>>(w.moff, bpm, sys->x, sys->y, sys->z, w.extra_xyzm, C,
                                                               j, R, w.key_a);
                count_launch(c);
                uint64_t *sk;
                int *si;
                if ((r = radix_sort(c, sys->n, 1, &sk, &si, s, true)) != RV_OK) return r;
                sel_member_write_k<<<M, 256, 0, s>>>(w.moff, sk, si, cap, C, j, w.lb + kLbGaveUp,
                                                     w.pert_idx, w.npert, w.st);
                count_launch(c);
            }
        }
    } else if (chain) {
        cudaMemsetAsync(w.npert, 0, sizeof(int) * NC, s);
    }
    if (quad) {
        cudaMemsetAsync(w.pflag, 0, (size_t)std::max<int64_t>(sys->n, 1), s);
        mark_pert_k<<<dim3(ceil_div(cap, 128), NC), 128, 0, s>>>(cap, w.pert_idx, w.npert, w.pflag);
        count_launch(c);
    }
    if ((r = build_tree(c, M, off, sys->x, sys->y, sys->z, sys->m, s)) != RV_OK) return r;
    const uint8_t *gact = nullptr;
    if (blk) {
        launch_block_groups(c, *blk, s);
        gact = w.gact;
    }
    // relative criterion (cfg.mac = 1): the accelerations in the system arrays (the previous
    // pass's, zero before the first one) are the references, read before they are overwritten
    const RelMac rel{c->cfg.alpha, sys->ax, sys->ay, sys->az};
    if ((r = tree_walk(c, c->cfg.theta, c->cfg.eps_star, NC, w.extra_xyzm, w.extra_eps, nullptr, C,
                       sys->ax, sys->ay, sys->az, sys->pot, w.extra_out, s, nullptr,
                       c->cfg.mac == 1 ? &rel : nullptr, gact, quad ? w.extra_quad : nullptr,
                       quad ? w.pflag : nullptr)) != RV_OK)
        return r;
    c->pert_members = NC;
    if (chain) {
        gather_pert_k<<<dim3(ceil_div(cap, 128), NC), 128, 0, s>>>(cap, w.pert_idx, w.npert, sys->x, sys->y, sys->z,
                                                                  sys->m, w.pert_m, w.pert_x);
        count_launch(c);
        ChainView V{sys->n_chain, cap, sys->chain_m, sys->chain_x, w.npert, w.pert_m, w.pert_x};
        r = coupling(c, NC, V, w.pert_a, w.pert_pot, w.chain_ext_a, w.chain_ext_pot, w.out8, s);
        if (r != RV_OK) return r;
        apply_pert_k<<<dim3(ceil_div(cap, 128), NC), 128, 0, s>>>(cap, w.pert_idx, w.npert, w.pert_a, w.pert_pot,
                                                                 sys->ax, sys->ay, sys->az, sys->pot,
                                                                 blk ? blk->level : nullptr, blk ? blk->n : 0,
                                                                 blk ? blk->L : 0);
        count_launch(c);
        chain_accel_k<<<ceil_div(NC * sys->n_chain, 128), 128, 0, s>>>(NC, sys->n_chain, sys->chain_m, sys->chain_x,
                                                                      w.chain_ext_a, w.chain_ext_pot, w.extra_out,
                                                                      w.out8, sys->chain_a, sys->chain_pot);
        count_launch(c);
    }
    return cuda_check(c, cudaGetLastError(), "system forces");
}

// ---------------------------------------------------------------------------
// kick-drift-kick
// ---------------------------------------------------------------------------
__global__ void kick_drift_k(int64_t n, float *x, float *y, float *z, float *vx, float *vy, float *vz,
                             const float *ax, const float *ay, const float *az, float hdt, float dt, int drift) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float u = fmaf(ax[i], hdt, vx[i]), v = fmaf(ay[i], hdt, vy[i]), w = fmaf(az[i], hdt, vz[i]);
        vx[i] = u; vy[i] = v; vz[i] = w;
        if (drift) {
            x[i] = fmaf(u, dt, x[i]); y[i] = fmaf(v, dt, y[i]); z[i] = fmaf(w, dt, z[i]);
        }
    }
}

__global__ void chain_kick_drift_k(int n, double *cx, double *cv, const double *ca, double hdt, double dt, int drift) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x)
        for (int a = 0; a < 3; a++) {
            cv[3 * k + a] += ca[3 * k + a] * hdt;
            if (drift) cx[3 * k + a] += cv[3 * k + a] * dt;
        }
}

void kick(rv_ctx *c, rv_system *sys, double dt, int drift, cudaStream_t s) {
    if (sys->n > 0) {
        kick_drift_k<<<grid_n(c, sys->n), 256, 0, s>>>(sys->n, sys->x, sys->y, sys->z, sys->vx, sys->vy, sys->vz,
                                                      sys->ax, sys->ay, sys->az, (float)(0.5 * dt), (float)dt, drift);
        count_launch(c);
    }
    if (sys->n_chain > 0) {
        const int nc = system_chains(sys) * sys->n_chain;
        chain_kick_drift_k<<<ceil_div(nc, 128), 128, 0, s>>>(nc, sys->chain_x, sys->chain_v, sys->chain_a, 0.5 * dt, dt,
                                                             drift);
        count_launch(c);
    }
}

rv_status kdk(rv_ctx *c, rv_system *sys, double dt, int nsteps, cudaStream_t s) {
    for (int step = 0; step < nsteps; step++) {
        kick(c, sys, dt, 1, s);
        rv_status r = system_forces(c, sys, s);
        if (r != RV_OK) return r;
        kick(c, sys, dt, 0, s);
    }
    return cuda_check(c, cudaGetLastError(), "kdk");
}

// ---------------------------------------------------------------------------
// FP64 totals per member: fixed grid, fixed per-thread striding, fixed tree
// reductions, so the result does not depend on scheduling
// ---------------------------------------------------------------------------
constexpr int kRedQ = 9;  // ekin, epot, P(3), L(3), mass

static int energy_bpm(int M) { return std::max(1, std::min(256, kRedSlots / M)); }

// Tree sums of kRedQ rows of 256 (o = 128 .. 1, element t + o onto t) into column
// 0: the strides below a warp by shuffles, one row a warp, the same pairs.
__device__ __forceinline__ void red_tree(double (*sm)[256]) {
    for (int o = 128; o >= 32; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int a = 0; a < kRedQ; a++) sm[a][threadIdx.x] += sm[a][threadIdx.x + o];
        __syncthreads();
    }
    for (int a = threadIdx.x >> 5; a < kRedQ; a += 8) {
        double s = sm[a][threadIdx.x & 31];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) sm[a][0] = s;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256) energy_partial_k(const int64_t *moff, int bpm, const float *x, const float *y,
                                                        const float *z, const float *vx, const float *vy,
                                                        const float *vz, const float *m, const float *pot,
                                                        double *part) {
    __shared__ double sm[kRedQ][256];
    const int mb = blockIdx.y;
    double q[kRedQ] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int64_t i = moff[mb] + (int64_t)blockIdx.x * 256 + threadIdx.x; i < moff[mb + 1]; i += (int64_t)bpm * 256) {
        double mi = m[i], X = x[i], Y = y[i], Z = z[i], U = vx[i], V = vy[i], W = vz[i];
        q[0] += 0.5 * mi * (U * U + V * V + W * W);
        q[1] += 0.5 * mi * (double)pot[i];
        q[2] += mi * U; q[3] += mi * V; q[4] += mi * W;
        q[5] += mi * (Y * W - Z * V); q[6] += mi * (Z * U - X * W); q[7] += mi * (X * V - Y * U);
        q[8] += mi;
    }
    for (int a = 0; a < kRedQ; a++) sm[a][threadIdx.x] = q[a];
    __syncthreads();
    red_tree(sm);
    if (threadIdx.x < kRedQ) part[kRedQ * ((int64_t)mb * bpm + blockIdx.x) + threadIdx.x] = sm[threadIdx.x][0];
}

__global__ void __launch_bounds__(256) energy_final_k(const double *part, int bpm, int n_ch, const double *cm,
                                                      const double *cx, const double *cv, const double *cpot,
                                                      double *out) {
    __shared__ double sm[kRedQ][256];
    const int mb = blockIdx.x;
    for (int a = 0; a < kRedQ; a++)
        sm[a][threadIdx.x] = ((int)threadIdx.x < bpm) ? part[kRedQ * ((int64_t)mb * bpm + threadIdx.x) + a] : 0.0;
    __syncthreads();
    red_tree(sm);
    if (threadIdx.x == 0) {
        double q[kRedQ];
        for (int a = 0; a < kRedQ; a++) q[a] = sm[a][0];
        for (int k = 0; k < n_ch; k++) {
            const int64_t kk = (int64_t)mb * n_ch + k;
            double mk = cm[kk];
            const double *X = cx + 3 * kk, *V = cv + 3 * kk;
            q[0] += 0.5 * mk * (V[0] * V[0] + V[1] * V[1] + V[2] * V[2]);
            q[1] += 0.5 * mk * cpot[kk];
            q[2] += mk * V[0]; q[3] += mk * V[1]; q[4] += mk * V[2];
            q[5] += mk * (X[1] * V[2] - X[2] * V[1]);
            q[6] += mk * (X[2] * V[0] - X[0] * V[2]);
            q[7] += mk * (X[0] * V[1] - X[1] * V[0]);
            q[8] += mk;
        }
        double *o = out + 10 * (int64_t)mb;
        o[0] = q[0]; o[1] = q[1]; o[2] = q[0] + q[1];
        for (int a = 0; a < 6; a++) o[3 + a] = q[2 + a];
        o[9] = q[8];
    }
}

rv_status energy(rv_ctx *c, const rv_system *sys, double *out, cudaStream_t s) {
    const int M = system_members(sys);
    int64_t tmp[2];
    rv_status r = upload_offsets(c, M, system_offsets(sys, tmp), s);
    if (r != RV_OK) return r;
    const int bpm = energy_bpm(M);
    energy_partial_k<<<dim3(bpm, M), 256, 0, s>>>(c->w.moff, bpm, sys->x, sys->y, sys->z, sys->vx, sys->vy, sys->vz,
                                                  sys->m, sys->pot, c->w.red);
    count_launch(c);
    // chain members of member m: the n_chains chains of that member, one after another
    energy_final_k<<<M, 256, 0, s>>>(c->w.red, bpm, sys->n_chain > 0 ? chains_per_member(sys) * sys->n_chain : 0,
                                     sys->chain_m, sys->chain_x, sys->chain_v, sys->chain_pot, out);
    count_launch(c);
    return cuda_check(c, cudaGetLastError(), "energy");
}

// ---------------------------------------------------------------------------
// CUDA graph of one step (kick-drift-kick [+ energy]), captured once per
// (system, dt, energy output) and replayed
// ---------------------------------------------------------------------------
static unsigned long long graph_key(const rv_system *sys, double dt, const double *eout) {
    unsigned long long h = 1469598103934665603ull;
    const unsigned char *p = reinterpret_cast<const unsigned char *>(sys);
    for (size_t i = 0; i < sizeof(rv_system); i++) h = (h ^ p[i]) * 1099511628211ull;
    const int M = system_members(sys);
    if (sys->member_offsets)
        for (int k = 0; k <= M; k++) h = (h ^ (unsigned long long)sys->member_offsets[k]) * 1099511628211ull;
    unsigned long long d;
    memcpy(&d, &dt, sizeof d);
    h = (h ^ d) * 1099511628211ull;
    h = (h ^ (unsigned long long)(uintptr_t)eout) * 1099511628211ull;
    return h;
}

rv_status kdk_graph(rv_ctx *c, rv_system *sys, double dt, int nsteps, double *eout, cudaStream_t s) {
    const unsigned long long key = graph_key(sys, dt, eout);
    if (!c->graph || c->graph_key != key) {
        if (c->graph) {
            cudaGraphExecDestroy(c->graph);
            c->graph = nullptr;
        }
        // settle everything a capture must not do (offset upload, kernel attributes) with an uncaptured
        // force evaluation at the current positions, which the step's first kick already expects
        rv_status r = system_forces(c, sys, s);
        if (r != RV_OK) return r;
        if ((r = cuda_check(c, cudaStreamSynchronize(s), "graph prepare")) != RV_OK) return r;
        cudaGraph_t g = nullptr;
        if ((r = cuda_check(c, cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "begin capture")) != RV_OK)
            return r;
        const long long l0 = c->launches;
        r = kdk(c, sys, dt, 1, s);
        if (r == RV_OK && eout) r = energy(c, sys, eout, s);
        cudaError_t e = cudaStreamEndCapture(s, &g);
        if (r != RV_OK) {
            if (g) cudaGraphDestroy(g);
            return r;
        }
        if (e != cudaSuccess) return cuda_check(c, e, "end capture");
        cudaGraphExec_t ge = nullptr;
        e = cudaGraphInstantiate(&ge, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return cuda_check(c, e, "graph instantiate");
        c->graph = ge;
        c->graph_key = key;
        c->graph_skey = c->w.skey;
        c->graph_perm = c->w.perm;
        c->graph_launches = c->launches - l0;
        c->launches = l0;
    }
    if (nsteps > 0) {
        // another build on this context may have come since the capture: the captured kernels
        // read the member offsets from the workspace, and after the replay the tree in the
        // workspace is the captured step's
        const int M = system_members(sys);
        int64_t tmp[2];
        const int64_t *off = system_offsets(sys, tmp);
        rv_status r = upload_offsets(c, M, off, s);
        if (r != RV_OK) return r;
        c->n = sys->n;
        c->max_member = 0;
        for (int k = 0; k < M; k++) c->max_member = std::max<int64_t>(c->max_member, off[k + 1] - off[k]);
        c->w.skey = c->graph_skey;
        c->w.perm = c->graph_perm;
        c->pert_members = system_chains(sys);
        c->built = true;
    }
    for (int k = 0; k < nsteps; k++) {
        cudaError_t e = cudaGraphLaunch(c->graph, s);
        if (e != cudaSuccess) return cuda_check(c, e, "graph launch");
        c->launches += c->graph_launches;
    }
    return RV_OK;
}

}  // namespace rv

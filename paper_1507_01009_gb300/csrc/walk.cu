// walk.cu -- Barnes-Hut tree walk and interaction evaluation (FP32).
//
// One warp walks the tree for one group of up to 64 consecutive stars, or, in
// small builds, for one part of a group's walk (Part). Cells are tested up to 64
// a pass, two per lane, under the box-box opening test; accepted cells are
// staged in shared memory as multipole records, opened leaves stage their
// stars, opened internal cells push their child range on a per-warp stack.
// Whenever a staged list holds a full tile, the warp evaluates it: a lane holds two stars of the group (a target pair), each of
// the p = ceil(s / 2) pairs is served by k = floor(32 / p) lanes, lane t + i p
// taking list pairs i, i + k, ... with broadcast shared-memory reads and
// evaluating every loaded source pair on both its stars; tile sums are added
// to running totals with Neumaier compensation, and the k partial totals of a
// star are combined in lane order at the end. Particles outside the tree (a chain's
// centre of mass) are walked by the same kernel as one-star groups before the
// tree's own groups.
//
// Staged lists hold list entries in pairs, each field of the two entries
// side by side, so that one lane evaluates two interactions with the packed
// two-wide FP32 instructions (add/mul/fma .f32x2). Each interaction is still
// computed element by element in FP32 round-to-nearest; only the order of the
// running sums differs from one entry per instruction.
//
// Interactions (G = 1, Sect. 3 Plummer softening; multipoles about the cell's
// centre of mass, Sect. 1):
//   star j on star i:  a += m_j r / (r^2 + e^2)^{3/2},  phi -= m_j (r^2 + e^2)^{-1/2},  r = x_j - x_i
//   cell on star i:    r = x_i - com, rho^2 = r.r + e^2,
//                      a += -M r / rho^3 + Q r / rho^5 - 5 (r.Q.r) r / (2 rho^7),
//                      phi -= M / rho + (r.Q.r) / (2 rho^5).
// Flops per interaction in this source (add/mul 1, FMA 2, rsqrt 1):
//   star-star 20, cell (monopole + quadrupole) 54, cell (monopole) 18.
#include <algorithm>

#include "rv_internal.cuh"

// What bounds it: instruction dispatch. A packed FP32 instruction takes two
// dispatch cycles of its scheduler and every other instruction at least one
// (the evaluation loop alone, any number of warps from 8 an SM up, reaches 0.82
// of the FMA peak for cells and 0.71 for stars: 132 + ~27 and 52 + ~19 cycles an
// iteration), so a pass that tests, stages and evaluates is worth what its
// instructions add up to; on 2^20 stars at theta 0.5 the packed instructions
// are 75 % of the walk's dispatch cycles.
//
// Unrolling of the evaluation loops (list pairs in flight per lane, each on
// two targets; measured on GB300: star pairs 1, cell pairs 4, which also divides
// every tile) and the register budget of the walk kernel. The kernel runs one
// warp per block; 112 registers a thread (the running sums and what a work item
// needs at its end live in shared memory) give 16 warps per SM, as 104 and 128
// do, and 4 bytes spill. Walk of 2^20 stars at theta 0.5 / 2^22 at 0.8, tile 96:
// 8.44 / 18.2 ms at 112, 8.60 / 18.7 at 104, 9.07 / 19.7 at 120, 9.2 / 19.9 at
// 128; cell pairs 2, 3, 4, 6, 8 at 112: 8.86, 8.52, 8.44, 8.36, 8.36 ms, but 65536
// stars (short tiles, two copies of the loop in use) 541 us at 4, 570 at 6, 619 at 8.
// Under spline softening the loops carry a branch per pair and the code of an
// unrolled cell loop no longer stays in the instruction cache beside the star loop:
// cell pairs 1, 2, 3, 4 there take 11.01, 10.82, 10.99, 11.77 ms on 2^20 stars
// (theta 0.5, groups of 64), 11.63, 11.52, 12.30, 13.81 in groups of 32, 7.15, 7.86,
// 9.09, 10.01 under the relative criterion in groups of 32, and 1.14, 1.31, 1.54,
// 1.68 on 100003 stars; one it is.
#ifndef RV_P2P_UNROLL
#define RV_P2P_UNROLL 1
#endif
#ifndef RV_M2P_UNROLL
#define RV_M2P_UNROLL 4
#endif
#ifndef RV_M2P_UNROLL_SPLINE
#define RV_M2P_UNROLL_SPLINE 1
#endif
#ifndef RV_WALK_MAXNREG
#define RV_WALK_MAXNREG 112
#endif
#ifdef RV_WALK_MIN_BLOCKS
#define RV_WALK_BOUNDS __launch_bounds__(kWalkWarps * 32, RV_WALK_MIN_BLOCKS)
#else
#define RV_WALK_BOUNDS __maxnreg__(RV_WALK_MAXNREG)
#endif

namespace rv {

// spline softening lengths (h = 2.8 eps): h^2, 1/h, 1/h^3
struct Spline {
    float h2, hinv, hinv3;
};

struct WalkArgs {
    const float4 *pos;   // sorted (x, y, z, m)
    const int4 *cbox;
    const int4 *clink;   // (child first, child end, first star, end star)
    const float4 *cmom;  // relative to the cell's geometric centre
    const int4 *groups;
    const int *perm;
    DevState *st;
    int cell_cap;
    int n;               // stars of the tree
    const int64_t *moff; // member star offsets [M + 1]
    int M;               // members (independent systems)
    const double *mbounds;  // per member: min x, y, z, L, 2^21 / L
    const int *mroot;    // root cell of each member
    const int *xmem;     // member of each extra particle (nullptr: member 0)
    int extra_per_member;  // > 0: extras [m e, (m + 1) e) belong to member m (e chains per member)
    MacTable mac;
    float eps2;          // star-star and star-cell softening^2
    float eps_star;
    int tile;
    int n_extra;
    const float *xyzm;   // extra particles (x, y, z, m)
    const float *xeps;
    const float4 *xquad; // optional: each extra particle's traceless quadrupole, 2 float4 (see extra_terms)
    const uint8_t *xq_skip;  // optional, per star (caller order): 1 = no quadrupole terms (a chain's perturber)
    float *ax, *ay, *az, *pot;
    float *xout;
    // optional record of accepted (group, cell) pairs that a walk at the
    // smaller angle theta_rec would have opened (the learned correction's input)
    MacTable rec;
    int2 *pairs;
    int *npairs;
    int pair_cap;
    // relative opening criterion: tolerance and reference acceleration per star (caller order)
    float rel_alpha;
    const float *arx, *ary, *arz;
    // optional group mask (block time steps): only groups with gact[g] != 0 are walked
    const uint8_t *gact;
    // queue order of the work items (null: build order, `parts` items a group),
    // and the per-star list cost written for the next walk's order
    const int *order;
    const uint8_t *opart;
    float *scost;
    // parts of the groups' walks (Part)
    int parts, n_leaf;
    float4 *partial;   // [part][sums, compensations][sorted star]
    int *garrive;
    // spline softening of the stars (h = 2.8 eps)
    Spline spl;
    // the walk stack's entries beyond kStackSm: kStackSpill per warp of the launch
    int *gstack;
};

// Per-warp shared memory: stack | lf_delta[64] | cell staging | star staging |
// running sums. Cell staging: (tile + 64) / 2 pairs of multipole records, 5
// float4 per pair holding (M, cx), (cy, cz), (-Qxx, -Qyy), (-Qzz, -Qxy),
// (-Qxz, -Qyz) of both entries side by side (cx.. = centre of mass relative
// to the group centre). Star staging: (tile + 64) / 2 pairs, 2 float4 per
// pair: (x, y), (z, m). Running sums: 16 floats per lane (AccSm).
constexpr int kCellPairF4 = 5, kStarPairF4 = 2;
constexpr int kAccWords = 16 * 32;
constexpr int kP2PUnroll = RV_P2P_UNROLL, kM2PUnroll = RV_M2P_UNROLL, kM2PUnrollSpline = RV_M2P_UNROLL_SPLINE;
__host__ __device__ inline size_t warp_staging_bytes(int tile) {
    return (size_t)kStackSm * 4 + 64 * 4 + (size_t)(tile + 64) / 2 * 16 * kCellPairF4 +
           (size_t)(tile + 64) / 2 * 16 * kStarPairF4;
}
__host__ __device__ inline size_t warp_smem_bytes(int tile) { return warp_staging_bytes(tile) + 4 * kAccWords; }

// The tree of one member as the walk sees it.
struct TreeGeo {
    int ncell;           // cells of all trees (at most the workspace capacity)
    int root;            // the member's root cell (-1: empty member)
    float lo[3], unit;   // the member's bounding-cube corner and grid unit in FP32
};

__device__ __forceinline__ TreeGeo tree_geo(const WalkArgs &A, int member) {
    TreeGeo t;
    t.ncell = min(A.st->ncell, A.cell_cap);
    t.root = A.mroot[member];
    const double *b = A.mbounds + 5 * member;
    t.lo[0] = (float)b[0];
    t.lo[1] = (float)b[1];
    t.lo[2] = (float)b[2];
    t.unit = (float)(b[3] / 2097152.0);
    return t;
}

struct Acc {
    float ax, ay, az, ph;      // running sums
    float cx, cy, cz, cp;      // Neumaier compensation
};

// Two FP32 values in one 64-bit register (low half: the even list entry).
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 d;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 f2_pack(float lo, float hi) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float f2_sum(f2 v) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return lo + hi;
}
__device__ __forceinline__ f2 f2_rsqrt(f2 v, bool guard_zero) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    float a = rsqrtf(lo), b = rsqrtf(hi);
    if (guard_zero) {
        a = (lo > 0.f) ? a : 0.f;
        b = (hi > 0.f) ? b : 0.f;
    }
    return f2_pack(a, b);
}
constexpr f2 kF2MinusHalf = 0xBF000000BF000000ull;     // (-0.5f, -0.5f)
constexpr f2 kF2MinusFiveHalf = 0xC0200000C0200000ull; // (-2.5f, -2.5f)

// A lane's two targets (minus their positions relative to the group's
// centre, each in both halves) and its share of a staged list: pairs j0,
// j0 + k, ... (j0 >= 2^20: the lane takes no share). Both targets use every
// source pair the lane loads.
struct Tgt {
    f2 nx[2], ny[2], nz[2];
    int j0, k;
};

// A lane's running sums for its two targets, kept in the warp's shared memory
// (not registers, which the evaluation loops need): for target q the sums (ax,
// ay, az, ph) at float4 2 q * 32 + lane, their Neumaier compensations at (2 q +
// 1) * 32 + lane, so a tile's sums take eight 16-byte accesses of consecutive lanes.
struct AccSm {
    float4 *p;   // the warp's region + lane
};

__device__ __forceinline__ void add_tile(const AccSm &A, int q, f2 tx, f2 ty, f2 tz, f2 tp) {
    float4 s = A.p[2 * q * 32], c = A.p[(2 * q + 1) * 32];
    nadd(s.x, c.x, f2_sum(tx));
    nadd(s.y, c.y, f2_sum(ty));
    nadd(s.z, c.z, f2_sum(tz));
    nadd(s.w, c.w, -f2_sum(tp));
    A.p[2 * q * 32] = s;
    A.p[(2 * q + 1) * 32] = c;
}

// Spline softening (the "spline" option of Sect. 2): the point mass smoothed
// by the cubic spline kernel of support h = 2.8 eps, so that phi(0) = -m/eps
// as for Plummer softening of length eps. From the kernel's enclosed mass,
// a = m d f(u) / h^3 and phi = (m/h) P(u) with u = |d| / h:
//   u < 1/2:  f = 32/3 - 192/5 u^2 + 32 u^3,  P = -14/5 + 16/3 u^2 - 48/5 u^4 + 32/5 u^5
//   u < 1:    f = 64/3 - 48 u + 192/5 u^2 - 32/3 u^3 - 1/(15 u^3),
//             P = -16/5 + 1/(15 u) + 32/3 u^2 - 16 u^3 + 48/5 u^4 - 32/15 u^5
//   u >= 1:   Newton.


// m f / h^3 and -m P / h (the walk sums -phi) for one pair at squared distance r2 < h^2
__device__ __forceinline__ void spline_terms(float r2, float m, const Spline &S, float &mr3, float &mr) {
    const float u = sqrtf(r2) * S.hinv;
    const float u2 = u * u;
    float f, P;
    if (u < 0.5f) {
        f = fmaf(u2, fmaf(32.f, u, -192.f / 5.f), 32.f / 3.f);
        P = fmaf(u2, fmaf(u2, fmaf(32.f / 5.f, u, -48.f / 5.f), 16.f / 3.f), -14.f / 5.f);
    } else {
        const float iu = 1.f / u;
        f = fmaf(u2, fmaf(-32.f / 3.f, u, 192.f / 5.f), fmaf(-48.f, u, 64.f / 3.f)) - (1.f / 15.f) * (iu * iu * iu);
        P = fmaf(u2, fmaf(u, fmaf(u, fmaf(-32.f / 15.f, u, 48.f / 5.f), -16.f), 32.f / 3.f),
                 fmaf(1.f / 15.f, iu, -16.f / 5.f));
    }
    mr3 = m * f * S.hinv3;
    mr = -m * P * S.hinv;
}

// One packed pair of star-star terms under spline softening: Newton beyond h,
// the kernel's field inside (per element).
__device__ __forceinline__ void spline_pair(f2 r2, f2 m2, const Spline &S, f2 &mr, f2 &mr3) {
    float ra, rb, ma, mb;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(ra), "=f"(rb) : "l"(r2));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(ma), "=f"(mb) : "l"(m2));
    float o3[2], o1[2];
    const float rr[2] = {ra, rb}, mm[2] = {ma, mb};
#pragma unroll
    for (int h = 0; h < 2; h++) {
        if (rr[h] >= S.h2) {
            const float ri = rsqrtf(rr[h]);
            o1[h] = mm[h] * ri;
            o3[h] = o1[h] * (ri * ri);
        } else {
            spline_terms(rr[h], mm[h], S, o3[h], o1[h]);
        }
    }
    mr = f2_pack(o1[0], o1[1]);
    mr3 = f2_pack(o3[0], o3[1]);
}

// Star pairs 0 .. npair-1 of a staged star list on this lane's targets:
//   d = x_j - x_i, a += m_j d / (d.d + e^2)^{3/2}, phi -= m_j / (d.d + e^2)^{1/2}
// (SPL: the spline field instead).
template <bool SOFT, bool SPL>
__device__ __forceinline__ void eval_p2p(const float4 *src, int npair, const Tgt &t, f2 eps2, const Spline &S,
                                         const AccSm &A) {
    f2 tx[2] = {0, 0}, ty[2] = {0, 0}, tz[2] = {0, 0}, tp[2] = {0, 0};   // tp sums +m/r
#pragma unroll kP2PUnroll
    for (int j = t.j0; j < npair; j += t.k) {
        const ulonglong2 a = reinterpret_cast<const ulonglong2 *>(src)[2 * j];      // x, y
        const ulonglong2 b = reinterpret_cast<const ulonglong2 *>(src)[2 * j + 1];  // z, m
#pragma unroll
        for (int q = 0; q < 2; q++) {
            f2 dx = f2_add(a.x, t.nx[q]), dy = f2_add(a.y, t.ny[q]), dz = f2_add(b.x, t.nz[q]);
            f2 mr, mr3;
            if (SPL) {
                f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
                spline_pair(r2, b.y, S, mr, mr3);
            } else {
                f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_fma(dz, dz, eps2)));
                f2 rinv = f2_rsqrt(r2, !SOFT);
                mr = f2_mul(b.y, rinv);
                mr3 = f2_mul(mr, f2_mul(rinv, rinv));
            }
            tx[q] = f2_fma(mr3, dx, tx[q]);
            ty[q] = f2_fma(mr3, dy, ty[q]);
            tz[q] = f2_fma(mr3, dz, tz[q]);
            tp[q] = f2_add(tp[q], mr);
        }
    }
    add_tile(A, 0, tx[0], ty[0], tz[0], tp[0]);
    add_tile(A, 1, tx[1], ty[1], tz[1], tp[1]);
}

// Cell pairs 0 .. npair-1 of a staged cell list on this lane's targets. With
// d = com - x_i = -r, rho^2 = d.d + e^2, the staged -Q gives q = -Q d = Q r
// and s = d.q / rho^4 = -(r.Q.r) / rho^4, so that
//   a += (M - 5/2 s) d / rho^3 + q / rho^5,  phi -= (M - s/2) / rho,
// which is the monopole + quadrupole expansion of the file header. SPL: the
// unsoftened expansion (e = 0), and a cell closer than h acts as the spline
// monopole.
template <bool QUAD, bool SPL>
__device__ __forceinline__ void eval_m2p(const float4 *src, int npair, const Tgt &t, f2 eps2, const Spline &S,
                                         const AccSm &A) {
    f2 tx[2] = {0, 0}, ty[2] = {0, 0}, tz[2] = {0, 0}, tp[2] = {0, 0};   // tp sums +(M - s/2)/rho
    if (SPL) eps2 = 0;
#pragma unroll(SPL ? kM2PUnrollSpline : kM2PUnroll)
    for (int j = t.j0; j < npair; j += t.k) {
        const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(src) + kCellPairF4 * j;
        const ulonglong2 a = p[0];   // M, cx
        const ulonglong2 b = p[1];   // cy, cz
        ulonglong2 c = make_ulonglong2(0, 0), e = c, f = c;
        if (QUAD) {
            c = p[2];   // -Qxx, -Qyy
            e = p[3];   // -Qzz, -Qxy
            f = p[4];   // -Qxz, -Qyz
        }
#pragma unroll
        for (int q = 0; q < 2; q++) {
            f2 dx = f2_add(a.y, t.nx[q]), dy = f2_add(b.x, t.ny[q]), dz = f2_add(b.y, t.nz[q]);
            f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_fma(dz, dz, eps2)));
            // r > 0: an accepted cell's box is separated from the group's box
            f2 rinv = f2_rsqrt(r2, false);
            f2 u = f2_mul(rinv, rinv);
            f2 rinv3 = f2_mul(rinv, u);
            f2 ix, iy, iz, ip;   // this pair's terms
            if (QUAD) {
                f2 qx = f2_fma(c.x, dx, f2_fma(e.y, dy, f2_mul(f.x, dz)));
                f2 qy = f2_fma(e.y, dx, f2_fma(c.y, dy, f2_mul(f.y, dz)));
                f2 qz = f2_fma(f.x, dx, f2_fma(f.y, dy, f2_mul(e.x, dz)));
                f2 dq = f2_fma(dx, qx, f2_fma(dy, qy, f2_mul(dz, qz)));
                f2 sw = f2_mul(dq, f2_mul(u, u));
                f2 rinv5 = f2_mul(rinv3, u);
                f2 B = f2_mul(rinv3, f2_fma(kF2MinusFiveHalf, sw, a.x));
                if (!SPL) {
                    tx[q] = f2_fma(B, dx, f2_fma(rinv5, qx, tx[q]));
                    ty[q] = f2_fma(B, dy, f2_fma(rinv5, qy, ty[q]));
                    tz[q] = f2_fma(B, dz, f2_fma(rinv5, qz, tz[q]));
                    tp[q] = f2_fma(rinv, f2_fma(kF2MinusHalf, sw, a.x), tp[q]);
                    continue;
                }
                ix = f2_fma(B, dx, f2_mul(rinv5, qx));
                iy = f2_fma(B, dy, f2_mul(rinv5, qy));
                iz = f2_fma(B, dz, f2_mul(rinv5, qz));
                ip = f2_mul(rinv, f2_fma(kF2MinusHalf, sw, a.x));
            } else {
                f2 mr3 = f2_mul(a.x, rinv3);
                if (!SPL) {
                    tx[q] = f2_fma(mr3, dx, tx[q]);
                    ty[q] = f2_fma(mr3, dy, ty[q]);
                    tz[q] = f2_fma(mr3, dz, tz[q]);
                    tp[q] = f2_fma(a.x, rinv, tp[q]);
                    continue;
                }
                ix = f2_mul(mr3, dx);
                iy = f2_mul(mr3, dy);
                iz = f2_mul(mr3, dz);
                ip = f2_mul(a.x, rinv);
            }
            if (SPL) {
                float ra, rb;
                asm("mov.b64 {%0, %1}, %2;" : "=f"(ra), "=f"(rb) : "l"(r2));
                if (ra < S.h2 || rb < S.h2) {   // a cell closer than h: the spline monopole
                    float m0, m1, o3, o1;
                    asm("mov.b64 {%0, %1}, %2;" : "=f"(m0), "=f"(m1) : "l"(a.x));
                    float v[4][2];
                    const f2 in4[4] = {ix, iy, iz, ip};
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(v[k][0]), "=f"(v[k][1]) : "l"(in4[k]));
                    float dd[3][2];
                    const f2 d3[3] = {dx, dy, dz};
#pragma unroll
                    for (int k = 0; k < 3; k++)
                        asm("mov.b64 {%0, %1}, %2;" : "=f"(dd[k][0]), "=f"(dd[k][1]) : "l"(d3[k]));
                    const float rr[2] = {ra, rb}, mm[2] = {m0, m1};
#pragma unroll
                    for (int hh = 0; hh < 2; hh++) {
                        if (rr[hh] < S.h2) {
                            spline_terms(rr[hh], mm[hh], S, o3, o1);
                            v[0][hh] = o3 * dd[0][hh];
                            v[1][hh] = o3 * dd[1][hh];
                            v[2][hh] = o3 * dd[2][hh];
                            v[3][hh] = o1;
                        }
                    }
                    ix = f2_pack(v[0][0], v[0][1]);
                    iy = f2_pack(v[1][0], v[1][1]);
                    iz = f2_pack(v[2][0], v[2][1]);
                    ip = f2_pack(v[3][0], v[3][1]);
                }
                tx[q] = f2_add(tx[q], ix);
                ty[q] = f2_add(ty[q], iy);
                tz[q] = f2_add(tz[q], iz);
                tp[q] = f2_add(tp[q], ip);
            }
        }
    }
    add_tile(A, 0, tx[0], ty[0], tz[0], tp[0]);
    add_tile(A, 1, tx[1], ty[1], tz[1], tp[1]);
}

// Field f of staged entry e in a pair-interleaved list whose pairs are
// `pair_f4` float4 long.
__device__ __forceinline__ float *staged(float4 *base, int pair_f4, int e, int f) {
    return reinterpret_cast<float *>(base + pair_f4 * (e >> 1)) + 2 * f + (e & 1);
}

// An odd list gets a massless partner in its last pair at the position of
// the entry beside it (finite, nonzero distance; contributes exactly 0).
__device__ __forceinline__ void pad_cells(float4 *m2p, int cnt) {
    if ((cnt & 1) && (threadIdx.x & 31) == 0) {
        float *d = reinterpret_cast<float *>(m2p + kCellPairF4 * (cnt >> 1));
        d[1] = 0.f;
        d[3] = d[2]; d[5] = d[4]; d[7] = d[6];
        for (int f = 4; f < 10; f++) d[2 * f + 1] = 0.f;
    }
}
__device__ __forceinline__ void pad_stars(float4 *p2p, int cnt) {
    if ((cnt & 1) && (threadIdx.x & 31) == 0) {
        float *d = reinterpret_cast<float *>(p2p + kStarPairF4 * (cnt >> 1));
        d[1] = d[0]; d[3] = d[2]; d[5] = d[4];
        d[7] = 0.f;
    }
}

__device__ __forceinline__ unsigned gap1(int blo, int bhi, int clo, int chi) {
    return (unsigned)max(max(clo - bhi, blo - chi), 0);
}

// The `mv` (<= 32) pairs from pair `from` on to the front of a staged list, field
// by field. Source and destination overlap when from < mv (tiles below 64
// entries): then every read of a field before its writes.
template <int F4>
__device__ __forceinline__ void move_front(float4 *list, int from, int mv) {
    const int lane = threadIdx.x & 31;
    const float4 *src = list + F4 * (from + lane);
    float4 *dst = list + F4 * lane;
    if (from >= 32) {
        if (lane < mv) {
#pragma unroll
            for (int f = 0; f < F4; f++) dst[f] = src[f];
        }
    } else {
        for (int f = 0; f < F4; f++) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lane < mv) v = src[f];
            __syncwarp();
            if (lane < mv) dst[f] = v;
            __syncwarp();
        }
    }
    __syncwarp();
}

// A work item's share of its group's walk: part q of P (P a power of two, pm =
// P - 1). Cells of more than `big` stars are traversed by every part; a cell at
// or below that size reached from a bigger one belongs, with everything under
// it, to part (its first star within its member) mod P, and so does every bigger
// cell that is accepted or is a leaf. The split depends on P and the member's
// tree alone, so a group's sums do not depend on which warps walk its parts, on
// the order they finish in or on a group mask. own = (part + member's first
// star) mod P; P = 1: pm = 0, own = 0, big = -1.
struct Part {
    int own, pm, big;
};

// Walks one part of the tree for one group; returns false if a bound was violated.
// Positions in the walk are relative to g, the geometric centre of the
// group's box: targets and staged sources are shifted once, cell centres of
// mass are (cell centre - g) + (centre of mass - cell centre). Differences of
// nearby FP32 coordinates are exact, so FP32 keeps its relative precision at
// any distance from the origin.
template <bool SOFT, bool QUAD, bool REC, bool REL, bool SPL>
__device__ __forceinline__ bool walk_group(const WalkArgs &A, const TreeGeo &G, const unsigned long long *thr,
                                           const unsigned long long *thr_rec, int gid, char *wsm, const int blo[3],
                                           const int bhi[3], const float g[3], const Tgt &tg, f2 eps2, const AccSm &acc,
                                           const Part &part, unsigned &np2p, unsigned &nm2p, float K) {
    const int lane = threadIdx.x & 31;
    const int T = A.tile;
    // the range stack: entries below kStackSm in shared memory, the deeper ones
    // (rare: a pass pushes at most 64, and the walk is depth-first) in this
    // warp's spill area in global memory; __syncwarp orders both for the warp.
    // An entry is a child range (first << 4 | owned << 3 | count - 1); `owned`:
    // the part owns everything under it.
    int *stack = reinterpret_cast<int *>(wsm);
    const unsigned spill0 = (blockIdx.x * kWalkWarps + (threadIdx.x >> 5)) * kStackSpill - kStackSm;
    static_assert((size_t)kStackSpillWarps * kStackSpill < 1u << 31, "32-bit spill offsets");
    int *lf_delta = stack + kStackSm;   // a pass's opened leaves: first star minus its place among the pass's stars
    float4 *m2p = reinterpret_cast<float4 *>(lf_delta + 64);
    float4 *p2p = m2p + kCellPairF4 * ((T + 64) / 2);
    const unsigned lt = lanemask_lt(), le = (lt << 1) | 1u;
    const int ncell = G.ncell;

    if (lane == 0) stack[0] = G.root << 4;  // the member's root: a range of one cell
    int top = 1, nm = 0, np = 0, hwm = 1;
    bool ok = true;
    // every pass tests at least one new cell, so a walk ends within ncell passes
    int guard = ncell + 1;
    __syncwarp();
    // a cell's records, opening test and link check (one of a pass's two slots per lane)
    struct Slot {
        int c;
        bool owned, accept, leaf, open, band;
        int4 lk, b;
        float4 r0, q1;
        float2 q2;
    };
    auto load_slot = [&](Slot &x) {
        // every record of the cell at once: one L2 round trip per pass. A slot
        // without a cell (c < 0), or with a bad index, reads the first or last cell's.
        const int c = min(max(x.c, 0), ncell - 1);
        x.b = __ldg(&A.cbox[c]);
        x.lk = __ldg(&A.clink[c]);
        x.r0 = __ldg(&A.cmom[3 * c + 0]);
        if (QUAD) {
            x.q1 = __ldg(&A.cmom[3 * c + 1]);
            x.q2 = __ldg(reinterpret_cast<const float2 *>(&A.cmom[3 * c + 2]));
        }
    };
    auto test_slot = [&](Slot &x) -> bool {   // returns "bad link"
        x.accept = x.leaf = x.open = x.band = false;
        bool bad = x.c >= ncell;
        if (x.c >= 0) {
            const int4 b = x.b;
            const int side = 1 << (kMaxLevel - b.w);
            const unsigned gx = gap1(blo[0], bhi[0], b.x, b.x + side);
            const unsigned gy = gap1(blo[1], bhi[1], b.y, b.y + side);
            const unsigned gz = gap1(blo[2], bhi[2], b.z, b.z + side);
            const unsigned long long d2 = (unsigned long long)gx * gx + (unsigned long long)gy * gy +
                                          (unsigned long long)gz * gz;
            if (REL && K >= 0.f) {
                // relative criterion: the group's box outside the cell's box grown by
                // side/10 per side (integers x 10), and M s^2 <= (K d^2) d^2 in FP32
                const int bo[3] = {b.x, b.y, b.z};
                bool outside = false;
#pragma unroll
                for (int a = 0; a < 3; a++)
                    outside |= (10 * bhi[a] <= 10 * bo[a] - side) || (10 * blo[a] >= 10 * (bo[a] + side) + side);
                const float d2f = __ull2float_rn(d2);
                const float s2 = __fmul_rn((float)side, (float)side);
                x.accept = outside && (__fmul_rn(x.r0.x, s2) <= __fmul_rn(__fmul_rn(K, d2f), d2f));
            } else {
                x.accept = d2 >= thr[b.w];
            }
            const bool mine = x.owned || ((x.lk.z & part.pm) == part.own);
            if (x.accept) {
                if (REC) x.band = mine && d2 < thr_rec[b.w];
                x.accept = mine;
            } else if (x.lk.x == x.lk.y) {
                x.leaf = mine;
                // links must stay inside the tree (a violated bound ends the walk with an error)
                bad |= (unsigned)x.lk.w > (unsigned)A.n || (unsigned)x.lk.z > (unsigned)x.lk.w;
            } else {
                // (a range's end is checked cell by cell, when they are popped)
                bad |= x.lk.x <= x.c || (unsigned)(x.lk.y - x.lk.x) > 8u;
                const bool shared = !x.owned && x.lk.w - x.lk.z > part.big;
                x.open = shared || mine;
                x.owned = !shared;   // of the children
            }
        }
        return bad;
    };
    auto stage_cell = [&](const Slot &x, int p) {
        float c0[3];
        geo_centre(x.b, G.lo, G.unit, c0);
        *staged(m2p, kCellPairF4, p, 0) = x.r0.x;
        *staged(m2p, kCellPairF4, p, 1) = (c0[0] - g[0]) + x.r0.y;
        *staged(m2p, kCellPairF4, p, 2) = (c0[1] - g[1]) + x.r0.z;
        *staged(m2p, kCellPairF4, p, 3) = (c0[2] - g[2]) + x.r0.w;
        if (QUAD) {   // q1 = (Qxx, Qyy, Qzz, Qxy), q2 = (Qxz, Qyz, 0, 0)
            *staged(m2p, kCellPairF4, p, 4) = -x.q1.x;
            *staged(m2p, kCellPairF4, p, 5) = -x.q1.y;
            *staged(m2p, kCellPairF4, p, 6) = -x.q1.z;
            *staged(m2p, kCellPairF4, p, 7) = -x.q1.w;
            *staged(m2p, kCellPairF4, p, 8) = -x.q2.x;
            *staged(m2p, kCellPairF4, p, 9) = -x.q2.y;
        }
    };
    auto push = [&](int p, const Slot &x) {
        const int e = (x.lk.x << 4) | (x.owned ? 8 : 0) | (x.lk.y - x.lk.x - 1);
        if (p < kStackSm) stack[p] = e;
        else if (p < kStackCap) A.gstack[spill0 + p] = e;
    };
    while (top > 0) {
        if (--guard < 0) { ok = false; break; }
        // pop whole child ranges from the top while they fit in the pass's 64
        // slots (slot s: lane s % 32, its first or second cell). Lane i holds
        // ranges i and i + 32 from the top; both prefix sums of their lengths run
        // in one register (16 bits each), and a slot finds its range from the
        // 64-bit mask of the ranges' first slots: its rank is the number of ranges
        // starting at or before it (a warp OR and a population count, instead of
        // writing the cells to shared memory and reading them back).
        const int avail = min(top, 64);
        const int i0 = top - 1 - lane, i1 = top - 33 - lane;
        int e0 = stack[min(max(i0, 0), kStackSm - 1)], e1 = stack[min(max(i1, 0), kStackSm - 1)];
        if (top > kStackSm) {
            if (i0 >= kStackSm) e0 = A.gstack[spill0 + i0];
            if (i1 >= kStackSm) e1 = A.gstack[spill0 + i1];
        }
        const int n0 = (lane < avail) ? (e0 & 7) + 1 : 0, n1 = (lane + 32 < avail) ? (e1 & 7) + 1 : 0;
        unsigned in = (unsigned)n0 | ((unsigned)n1 << 16);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, in, o);
            if (lane >= o) in += y;
        }
        const int in0 = in & 0xffff, in1 = (in >> 16) + (__shfl_sync(0xffffffffu, in, 31) & 0xffff);
        const bool fit0 = n0 > 0 && in0 <= 64, fit1 = n1 > 0 && in1 <= 64;
        const int s0 = in0 - n0, s1 = in1 - n1;
        const unsigned mlo = __reduce_or_sync(0xffffffffu, (fit0 && s0 < 32 ? 1u << (s0 & 31) : 0u) |
                                                               (fit1 && s1 < 32 ? 1u << (s1 & 31) : 0u));
        const unsigned mhi = __reduce_or_sync(0xffffffffu, (fit0 && s0 >= 32 ? 1u << (s0 & 31) : 0u) |
                                                               (fit1 && s1 >= 32 ? 1u << (s1 & 31) : 0u));
        const int total = __reduce_max_sync(0xffffffffu, max(fit0 ? in0 : 0, fit1 ? in1 : 0));
        const int klo = __popc(mlo);
        top -= klo + __popc(mhi);
        Slot xa, xb;
        {
            const unsigned ma = mlo & le, mb = mhi & le;
            const int ra = __popc(ma) - 1, rb = klo + __popc(mb) - 1;   // ranks of the slots' ranges (slot 0 starts one)
            const int sa = 31 - __clz(ma), sb = mb ? 63 - __clz(mb) : 31 - __clz(mlo);
            const int ea = __shfl_sync(0xffffffffu, e0, ra);
            const int eb0 = __shfl_sync(0xffffffffu, e0, rb & 31), eb1 = __shfl_sync(0xffffffffu, e1, rb & 31);
            const int eb = rb < 32 ? eb0 : eb1;
            xa.c = (lane < total) ? (ea >> 4) + (lane - sa) : -1;
            xb.c = (lane + 32 < total) ? (eb >> 4) + (lane + 32 - sb) : -1;
            xa.owned = (ea & 8) != 0;
            xb.owned = (eb & 8) != 0;
        }
        load_slot(xa);
        load_slot(xb);
        const bool bad_a = test_slot(xa), bad_b = test_slot(xb);
        if (__any_sync(0xffffffffu, bad_a || bad_b)) { ok = false; break; }
        // opened internal cells: push their child ranges (slot order)
        const unsigned oma = __ballot_sync(0xffffffffu, xa.open), omb = __ballot_sync(0xffffffffu, xb.open);
        if (xa.open) push(top + __popc(oma & lt), xa);
        if (xb.open) push(top + __popc(oma) + __popc(omb & lt), xb);
        top += __popc(oma) + __popc(omb);
        hwm = max(hwm, top);
        if (top > kStackCap) { ok = false; break; }
        // accepted cells: stage their multipole records, centre of mass relative to g, -Q
        const unsigned ama = __ballot_sync(0xffffffffu, xa.accept), amb = __ballot_sync(0xffffffffu, xb.accept);
        if (xa.accept) stage_cell(xa, nm + __popc(ama & lt));
        if (xb.accept) stage_cell(xb, nm + __popc(ama) + __popc(amb & lt));
        nm += __popc(ama) + __popc(amb);
        nm2p += __popc(ama) + __popc(amb);
        if (REC) {
            const unsigned bma = __ballot_sync(0xffffffffu, xa.band), bmb = __ballot_sync(0xffffffffu, xb.band);
            if (bma | bmb) {
                int base = 0;
                if (lane == 0) base = atomicAdd(A.npairs, __popc(bma) + __popc(bmb));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (xa.band) {
                    const int p = base + __popc(bma & lt);
                    if (p < A.pair_cap) A.pairs[p] = make_int2(gid, xa.c);
                    else latch_err(A.st, kErrPairs);
                }
                if (xb.band) {
                    const int p = base + __popc(bma) + __popc(bmb & lt);
                    if (p < A.pair_cap) A.pairs[p] = make_int2(gid, xb.c);
                    else latch_err(A.st, kErrPairs);
                }
            }
        }
        // opened leaves: stage their stars relative to g, leaves in slot order
        // and stars in order within each (the order the tiles take them), 32
        // stars a round whichever leaves they come from, two rounds' loads in
        // flight; a star finds its leaf as a slot finds its range
        const unsigned lma = __ballot_sync(0xffffffffu, xa.leaf), lmb = __ballot_sync(0xffffffffu, xb.leaf);
        if (lma | lmb) {
            const int ca = xa.leaf ? xa.lk.w - xa.lk.z : 0, cb = xb.leaf ? xb.lk.w - xb.lk.z : 0;
            int ia, ib;
            if (__any_sync(0xffffffffu, max(ca, cb) > 2047)) {   // overfull leaves of the finest level
                ia = ca;
                ib = cb;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int ya = __shfl_up_sync(0xffffffffu, ia, o);
                    const int yb = __shfl_up_sync(0xffffffffu, ib, o);
                    if (lane >= o) {
                        ia += ya;
                        ib += yb;
                    }
                }
            } else {   // both sums below 2^16
                unsigned iab = (unsigned)ca | ((unsigned)cb << 16);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, iab, o);
                    if (lane >= o) iab += y;
                }
                ia = (int)(iab & 0xffff);
                ib = (int)(iab >> 16);
            }
            ib += __shfl_sync(0xffffffffu, ia, 31);
            const int total_stars = __shfl_sync(0xffffffffu, ib, 31);
            const int sa = xa.leaf ? ia - ca : -1, sb = xb.leaf ? ib - cb : -1;   // -1: no window holds it
            if (xa.leaf) lf_delta[__popc(lma & lt)] = xa.lk.z - sa;
            if (xb.leaf) lf_delta[__popc(lma) + __popc(lmb & lt)] = xb.lk.z - sb;
            __syncwarp();
            int before = -1;   // leaves that started before the window, minus one
            for (int base = 0; base < total_stars; base += 64) {
                float4 st2[2];
                int cc[2];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int w0 = base + 32 * h, idx = w0 + lane;
                    cc[h] = min(32, total_stars - w0);   // <= 0: no second round
                    const unsigned m = __reduce_or_sync(
                        0xffffffffu, ((unsigned)(sa - w0) < 32u && sa >= 0 ? 1u << (sa - w0) : 0u) |
                                         ((unsigned)(sb - w0) < 32u && sb >= 0 ? 1u << (sb - w0) : 0u));
                    if (lane < cc[h]) st2[h] = __ldg(&A.pos[lf_delta[before + __popc(m & le)] + idx]);
                    before += __popc(m);
                }
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    if (lane < cc[h]) {
                        const int e = np + lane;
                        *staged(p2p, kStarPairF4, e, 0) = st2[h].x - g[0];
                        *staged(p2p, kStarPairF4, e, 1) = st2[h].y - g[1];
                        *staged(p2p, kStarPairF4, e, 2) = st2[h].z - g[2];
                        *staged(p2p, kStarPairF4, e, 3) = st2[h].w;
                    }
                    np += max(cc[h], 0);
                }
                // np < T before the two rounds, so at most T + 63 entries are ever staged
                while (np >= T) {
                    __syncwarp();
                    eval_p2p<SOFT, SPL>(p2p, T / 2, tg, eps2, A.spl, acc);
                    __syncwarp();
                    move_front<kStarPairF4>(p2p, T / 2, (np - T + 1) / 2);
                    np -= T;
                }
            }
            np2p += total_stars;
        }
        // a pass adds up to 64 cells: flush while a full tile is staged (nm < T
        // before every pass, so at most T + 63 entries are ever staged)
        while (nm >= T) {
            __syncwarp();
            eval_m2p<QUAD, SPL>(m2p, T / 2, tg, eps2, A.spl, acc);
            __syncwarp();
            move_front<kCellPairF4>(m2p, T / 2, (nm - T + 1) / 2);
            nm -= T;
        }
        __syncwarp();
    }
    __syncwarp();
    if (ok) {
        pad_stars(p2p, np);
        pad_cells(m2p, nm);
        __syncwarp();
        if (np > 0) eval_p2p<SOFT, SPL>(p2p, (np + 1) / 2, tg, eps2, A.spl, acc);
        if (nm > 0) eval_m2p<QUAD, SPL>(m2p, (nm + 1) / 2, tg, eps2, A.spl, acc);
    }
    __syncwarp();
    if (lane == 0) atomicMax(&A.st->stack_hwm, hwm);
    return ok;
}

// Zeroes the warp's running sums.
__device__ __forceinline__ void clear_acc(float4 *accw) {
#pragma unroll
    for (int k = 0; k < 4; k++) accw[32 * k + (threadIdx.x & 31)] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
}

// Lane l serves target pair t = l % p (stars 2t and 2t + 1) with share
// l / p; the k lanes t, t + p, ..., t + (k - 1) p of a pair add their partial
// totals in that order, read from the warp's running sums (AccSm). Returns the
// totals of stars `lane` and `lane + 32`.
__device__ __forceinline__ void combine_shares(const float4 *accw, int s, int p, int k, Acc out[2]) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int i = lane + 32 * h;   // star of the group
        Acc o = {};
        if (i < s)
            for (int m = 0; m < k; m++) {
                const float4 *e = accw + (i & 1) * 64 + (i >> 1) + m * p;
                const float4 v = e[0], w = e[32];
                nadd(o.ax, o.cx, v.x); nadd(o.ay, o.cy, v.y);
                nadd(o.az, o.cz, v.z); nadd(o.ph, o.cp, v.w);
                o.cx += w.x; o.cy += w.y; o.cz += w.z; o.cp += w.w;
            }
        out[h] = o;
    }
    __syncwarp();
}

// Direct terms of the extra particles of `member` on one target (pair
// softening rule of Sect. 3: max(eps_i, eps_j), none if either is
// unsoftened), absolute FP32. With A.xquad, an extra particle (a chain seen
// from outside) also carries a traceless quadrupole Q about its position,
// (xx, yy, zz, xy), (xz, yz, 0, 0), whose field is added as for a cell: with
// d = x_extra - x_i = -r and rho^2 = d.d + e^2,
//   a += -Q d / rho^5 + 5/2 (d.Q.d) d / rho^7,  phi -= (d.Q.d) / (2 rho^5),
// unless use_quad is false (a target that is a chain's perturber).
__device__ __forceinline__ void extra_terms(const WalkArgs &A, float xi, float yi, float zi, float ei, int skip,
                                            int member, Acc &acc, bool use_quad = true) {
    float tx = 0.f, ty = 0.f, tz = 0.f, tp = 0.f;
    const int k0 = A.extra_per_member ? member * A.extra_per_member : 0;
    const int k1 = A.extra_per_member ? min(k0 + A.extra_per_member, A.n_extra) : A.n_extra;
    for (int k = k0; k < k1; k++) {
        if (k == skip) continue;
        if (!A.extra_per_member && (A.xmem ? A.xmem[k] : 0) != member) continue;
        float ek = A.xeps[k];
        float e = (ei == 0.f || ek == 0.f) ? 0.f : fmaxf(ei, ek);
        float dx = A.xyzm[4 * k] - xi, dy = A.xyzm[4 * k + 1] - yi, dz = A.xyzm[4 * k + 2] - zi;
        float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, e * e)));
        if (r2 <= 0.f) continue;
        float rinv = rsqrtf(r2);
        float mr = A.xyzm[4 * k + 3] * rinv;
        float mr3 = mr * rinv * rinv;
        tx = fmaf(mr3, dx, tx); ty = fmaf(mr3, dy, ty); tz = fmaf(mr3, dz, tz);
        tp -= mr;
        if (A.xquad && use_quad) {
            const float4 q1 = A.xquad[2 * k], q2 = A.xquad[2 * k + 1];
            const float qx = fmaf(q1.x, dx, fmaf(q1.w, dy, q2.x * dz));
            const float qy = fmaf(q1.w, dx, fmaf(q1.y, dy, q2.y * dz));
            const float qz = fmaf(q2.x, dx, fmaf(q2.y, dy, q1.z * dz));
            const float dqd = fmaf(dx, qx, fmaf(dy, qy, dz * qz));
            const float u = rinv * rinv;
            const float r5 = rinv * u * u;
            const float b = 2.5f * dqd * r5 * u;
            tx = fmaf(b, dx, fmaf(-r5, qx, tx));
            ty = fmaf(b, dy, fmaf(-r5, qy, ty));
            tz = fmaf(b, dz, fmaf(-r5, qz, tz));
            tp = fmaf(-0.5f * dqd, r5, tp);
        }
    }
    nadd(acc.ax, acc.cx, tx); nadd(acc.ay, acc.cy, ty); nadd(acc.az, acc.cz, tz); nadd(acc.ph, acc.cp, tp);
}

// A part of a walk is done: nonzero in the warp that finishes the last of the P
// parts (whose sums every part has then written), which also resets the counter; 1 if
// every part's walk was whole, 2 if one was not (counted in the upper bits): then
// the group's stars get no forces, as when an unsplit walk ends early.
constexpr int kPartFailed = 1 << 16;
__device__ __forceinline__ int last_part(int *arrive, int P, bool ok) {
    int last = 0;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        __threadfence();   // this part's sums before its arrival
        const int old = atomicAdd(arrive, ok ? 1 : 1 + kPartFailed);
        if ((old & (kPartFailed - 1)) == P - 1) {
            last = ok && old < kPartFailed ? 1 : 2;
            *arrive = 0;
        }
        __threadfence();
    }
    last = __shfl_sync(0xffffffffu, last, 0);
    __syncwarp();   // the other parts' sums, acquired by lane 0, for every lane (a shuffle orders no memory)
    return last;
}

// A part's sums with their compensations (p: the part's slot of the star, `stride`
// between the two): a star's total is rounded once, however many parts it has. (The
// part with the star's own pair is of the size of m / eps, which the end takes out.)
__device__ __forceinline__ void put_part(float4 *p, int64_t stride, const Acc &t) {
    p[0] = make_float4(t.ax, t.ay, t.az, t.ph);
    p[stride] = make_float4(t.cx, t.cy, t.cz, t.cp);
}

// The parts' sums added in part order (p: the star's slot of the first part).
__device__ __forceinline__ Acc add_parts(const float4 *p, int64_t stride, int P) {
    Acc t = {};
    for (int q = 0; q < P; q++) {
        const float4 v = __ldcg(p + 2 * q * stride), w = __ldcg(p + (2 * q + 1) * stride);
        nadd(t.ax, t.cx, v.x); nadd(t.ay, t.cy, v.y); nadd(t.az, t.cz, v.z); nadd(t.ph, t.cp, v.w);
        t.cx += w.x; t.cy += w.y; t.cz += w.z; t.cp += w.w;
    }
    return t;
}

__device__ __forceinline__ Part part_of(int q, int P, int64_t m0, int64_t n_member, int n_leaf) {
    const int grain = (int)(n_member / kPartGrain);
    return Part{(int)((q + m0) & (P - 1)), P - 1, P > 1 ? max(n_leaf, grain) : -1};
}

// A work item of a group, as the warp keeps it in shared memory while it walks.
struct Item {
    int group, first, count, member, q, P;
};

// Work items: the extra particles (one-star groups whose box is their own grid
// cell [q, q+1)^3, q = floor((x - min) 2^21 / L) limited to +-2^23; never split:
// FP64 quantities are made from their forces), then the tree's groups in their parts.
template <bool SOFT, bool QUAD, bool REC, bool REL, bool SPL>
__global__ void RV_WALK_BOUNDS walk_tree_k(WalkArgs A) {
    extern __shared__ __align__(16) char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // per-level opening thresholds in shared memory: lanes of a warp test cells
    // of different levels, which a constant-bank read would serialise
    __shared__ unsigned long long mac_thr[kLevels];
    __shared__ unsigned long long rec_thr[REC ? kLevels : 1];
    __shared__ Item item[kWalkWarps];
    if (threadIdx.x < kLevels) mac_thr[threadIdx.x] = A.mac.thr[threadIdx.x];
    if (REC && threadIdx.x < kLevels) rec_thr[threadIdx.x] = A.rec.thr[threadIdx.x];
    __syncthreads();
    char *wsm = smem + wib * warp_smem_bytes(A.tile);
    const int nitem = A.n_extra + (A.order ? A.st->walk.nitem : max(A.st->ngroup, 0) * A.parts);
    while (true) {
        int gi = 0;
        if (lane == 0) gi = atomicAdd(&A.st->walk.next_item, 1);
        gi = __shfl_sync(0xffffffffu, gi, 0);
        if (gi >= nitem) break;
        float4 *accw = reinterpret_cast<float4 *>(wsm + warp_staging_bytes(A.tile));
        const AccSm acc{accw + lane};
        unsigned a2 = 0, a3 = 0;   // list entries of the group: stars, cells
        if (gi < A.n_extra) {
            // ---- a particle outside the tree: all 32 lanes share its interaction list
            // (both target slots hold it; the second slot's sums are not used)
            const int kx = gi;
            const int mk = A.extra_per_member ? kx / A.extra_per_member : (A.xmem ? A.xmem[kx] : 0);
            const TreeGeo G = tree_geo(A, mk);
            const double *mb = A.mbounds + 5 * mk;
            float xi = A.xyzm[4 * kx], yi = A.xyzm[4 * kx + 1], zi = A.xyzm[4 * kx + 2];
            float ek = A.xeps[kx];
            float e = (ek == 0.f || A.eps_star == 0.f) ? 0.f : fmaxf(ek, A.eps_star);
            int blo[3], bhi[3];
            const float pv[3] = {xi, yi, zi};
            for (int a = 0; a < 3; a++) {
                double q = floor(__dmul_rn(__dsub_rn((double)pv[a], mb[a]), mb[4]));
                q = fmin(fmax(q, -8388608.0), 8388608.0);
                blo[a] = (int)q;
                bhi[a] = (int)q + 1;
            }
            float g[3];
            geo_centre(make_int4(blo[0], blo[1], blo[2], kMaxLevel), G.lo, G.unit, g);
            Tgt tg;
            tg.nx[0] = tg.nx[1] = f2_pack(g[0] - xi, g[0] - xi);
            tg.ny[0] = tg.ny[1] = f2_pack(g[1] - yi, g[1] - yi);
            tg.nz[0] = tg.nz[1] = f2_pack(g[2] - zi, g[2] - zi);
            tg.j0 = lane;
            tg.k = 32;
            clear_acc(accw);
            bool ok = true;
            if (G.ncell > 0 && G.root >= 0)
                ok = walk_group<false, QUAD, false, false, false>(A, G, mac_thr, rec_thr, -1, wsm, blo, bhi, g, tg,
                                                           f2_pack(e * e, e * e), acc, Part{0, 0, -1}, a2, a3, -1.f);
            if (!ok) {
                if (lane == 0) latch_err(A.st, kErrStack);
                continue;
            }
            Acc tots[2];
            combine_shares(accw, 1, 1, 32, tots);
            Acc &tot = tots[0];
            if (lane == 0) {
                extra_terms(A, xi, yi, zi, ek, kx, mk, tot);
                A.xout[4 * kx] = tot.ax + tot.cx;
                A.xout[4 * kx + 1] = tot.ay + tot.cy;
                A.xout[4 * kx + 2] = tot.az + tot.cz;
                A.xout[4 * kx + 3] = tot.ph + tot.cp;
            }
            continue;
        }
        // ---- a part of a group's walk, in queue order (skipped when the mask says none of its stars is active)
        gi -= A.n_extra;
        const int gk = A.order ? A.order[gi] : gi / A.parts;
        if (A.gact && !A.gact[gk]) continue;
        const int q = A.order ? A.opart[gi] : gi % A.parts;
        const GroupRec grp = load_group(A.groups, gk);
        if (grp.first < 0 || grp.count < 1 || grp.count > kMaxGroup || grp.first + grp.count > A.n) {
            if (lane == 0) latch_err(A.st, kErrStack);
            continue;
        }
        Part part;
        TreeGeo G;
        {
            const int mg = member_of(A.moff, A.M, grp.first);
            const int P = parts_of_group(A.parts, grp.count);
            if (q >= P) continue;
            part = part_of(q, P, A.moff[mg], A.moff[mg + 1] - A.moff[mg], A.n_leaf);
            G = tree_geo(A, mg);
            __syncwarp();
            if (lane == 0) item[wib] = Item{gk, grp.first, grp.count, mg, q, P};
        }
        if (G.root < 0) {
            if (lane == 0) latch_err(A.st, kErrStack);
            continue;
        }
        const int *blo = grp.lo, *bhi = grp.hi;
        float g[3];
        box_centre(blo, bhi, G.lo, G.unit, g);
        // p target pairs (stars 2t, 2t + 1), k lanes per pair
        Tgt tg;
        {
            const int s = grp.count, p = (s + 1) >> 1, k = 32 / p;
            const int t = lane % p, sub = lane / p;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                // an odd group's last pair repeats its star; those sums are not used
                const float4 pq = __ldg(&A.pos[grp.first + min(2 * t + h, s - 1)]);
                // minus the star's position relative to g (exact: FP32 negation)
                const float nx = -(pq.x - g[0]), ny = -(pq.y - g[1]), nz = -(pq.z - g[2]);
                tg.nx[h] = f2_pack(nx, nx);
                tg.ny[h] = f2_pack(ny, ny);
                tg.nz[h] = f2_pack(nz, nz);
            }
            tg.j0 = (sub < k) ? sub : (1 << 20);  // lanes beyond k p take no list pairs
            tg.k = k;
        }
        // relative criterion: K = (alpha |a|min) u^2 of the group, as in the oracle;
        // a group without a reference (|a|min = 0, no force pass yet) walks at theta (K < 0)
        float K = -1.f;
        if (REL) {
            float am = __int_as_float(0x7f800000);
            for (int i = lane; i < grp.count; i += 32) {
                // |a| = sqrt((x x + y y) + z z) in FP32, one rounding per operation, as the oracle takes it
                const int j = A.perm[grp.first + i];
                const float x = A.arx[j], y = A.ary[j], z = A.arz[j];
                am = fminf(am, sqrtf(__fadd_rn(__fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y)), __fmul_rn(z, z))));
            }
            for (int o = 16; o > 0; o >>= 1) am = fminf(am, __shfl_xor_sync(0xffffffffu, am, o));
            if (am > 0.f) K = __fmul_rn(__fmul_rn(A.rel_alpha, am), __fmul_rn(G.unit, G.unit));
        }
        clear_acc(accw);
        const bool ok = walk_group<SOFT, QUAD, REC, REL, SPL>(A, G, mac_thr, rec_thr, gk, wsm, blo, bhi, g, tg,
                                                         f2_pack(A.eps2, A.eps2), acc, part, a2, a3, K);
        if (!ok && lane == 0) latch_err(A.st, kErrStack);
        // (what the end of the item needs is read again: the walk has no registers to keep it)
        const Item it = item[wib];
        const int s = it.count, p = (s + 1) >> 1, k = 32 / p, P = it.P, mg = it.member, first = it.first;
        if (ok && lane == 0) {
            atomicAdd(&A.st->walk.n_p2p, (unsigned long long)a2 * s);
            atomicAdd(&A.st->walk.n_m2p, (unsigned long long)a3 * s);
        }
        Acc tots[2];
        combine_shares(accw, s, p, k, tots);
        if (P > 1) {
            // the part's sums; the warp that finishes the group's last part adds
            // them up. Every part has read its stars' references by then.
            float4 *slot = A.partial + first;
#pragma unroll
            for (int h = 0; h < 2; h++)
                if (lane + 32 * h < s) put_part(slot + (int64_t)2 * it.q * A.n + lane + 32 * h, A.n, tots[h]);
            if (last_part(A.garrive + it.group, P, ok) != 1) continue;
#pragma unroll
            for (int h = 0; h < 2; h++)
                if (lane + 32 * h < s) tots[h] = add_parts(slot + lane + 32 * h, A.n, P);
        }
        if (!ok) continue;
        const float cost = P * ((float)a2 + 2.5f * (float)a3);   // list pairs, a cell costing ~2.5 stars
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int i = lane + 32 * h;
            if (i >= s) continue;
            Acc &tot = tots[h];
            const float4 ps = __ldg(&A.pos[first + i]);
            // the star's own pair was evaluated at r = 0: remove its -m/eps (the product
            // rounded on its own, as in the pair, so that the two cancel exactly)
            if (SOFT) tot.ph += __fmul_rn(ps.w, rsqrtf(A.eps2));
            int o = A.perm[first + i];
            if (A.n_extra > 0) extra_terms(A, ps.x, ps.y, ps.z, A.eps_star, -1, mg, tot, !(A.xq_skip && A.xq_skip[o]));
            A.ax[o] = tot.ax + tot.cx;
            A.ay[o] = tot.ay + tot.cy;
            A.az[o] = tot.az + tot.cz;
            A.pot[o] = tot.ph + tot.cp;
            A.scost[o] = cost;
        }
    }
}

// ---------------------------------------------------------------------------
// Queue order of the work items: most expensive first (longest-processing-time
// first: the walk's tail then holds the cheapest ones). The estimate is the
// list cost the last walk recorded for the group's first star, divided by the
// group's parts, if that walk covered the same number of stars (st->cost_n);
// otherwise the volume of the group's box, smallest first (small boxes sit in
// dense regions with long lists). Groups are bucketed by log2 of the estimate
// (1/16 steps), all parts of a group together; the order within a bucket is
// unspecified. The forces do not depend on it.
constexpr int kOrderBins = 1024;   // the workspace's obins holds this many
// Smaller systems walk their items in build order: the three launches cost more
// than the balance gives (walk of 16000 stars 150 us ordered or not, 65536 stars
// 562 -> 543 us, 100003 stars in groups of 32 957 -> 892 us).
constexpr int kOrderMinStars = 1 << 15;

struct OrderArgs {
    const int4 *groups;
    const int *perm;
    const float *scost;
    int parts, n;
};

__device__ __forceinline__ int order_bin(const OrderArgs &A, bool hist, int g, int &P) {
    const GroupRec r = load_group(A.groups, g);
    const int first = min(max(r.first, 0), A.n - 1);
    P = parts_of_group(A.parts, max(r.count, 1));
    float lv;
    if (hist) {
        // any stored value is a finite estimate >= 1 here (NaN -> 1)
        const float c = fminf(fmaxf(A.scost[A.perm[first]] / P, 1.f), 1e30f);
        lv = 64.f - log2f(c);   // descending cost (a cost above 2^64 shares the first bin)
    } else {
        lv = log2f((float)max(r.hi[0] - r.lo[0], 1)) + log2f((float)max(r.hi[1] - r.lo[1], 1)) +
             log2f((float)max(r.hi[2] - r.lo[2], 1));
    }
    return min(max((int)(16.f * lv), 0), kOrderBins - 1);
}

// (A) each group's bin (and its parts), and the bins' item counts (bins zeroed before)
__global__ void group_bins_k(OrderArgs A, const DevState *st, int *gbin, int *bins) {
    const int ng = st->ngroup;
    const bool hist = st->cost_n == A.n;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
        int P;
        const int b = order_bin(A, hist, g, P);
        gbin[g] = b * (2 * kMaxParts) + P;
        atomicAdd(&bins[b], P);
    }
}

// (B) exclusive scan of the bin counts, one bin per thread; the walk that
// follows records the costs of its stars
__global__ void __launch_bounds__(kOrderBins) group_bins_scan_k(DevState *st, int n, int *bins) {
    __shared__ int wsum[kOrderBins / 32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int v = bins[t];
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int x = wsum[lane];
        int sx = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, sx, o);
            if (lane >= o) sx += y;
        }
        wsum[lane] = sx - x;
    }
    __syncthreads();
    bins[t] = incl - v + wsum[w];
    if (t == kOrderBins - 1) st->walk.nitem = incl + wsum[w];
    if (t == 0) st->cost_n = n;
}

// (C) each group's items to the next free slots of its bin
__global__ void group_scatter_k(const DevState *st, const int *gbin, int *bins, int *order, uint8_t *opart) {
    const int ng = st->ngroup;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) {
        const int b = gbin[g], P = b % (2 * kMaxParts);
        const int at = atomicAdd(&bins[b / (2 * kMaxParts)], P);
        for (int q = 0; q < P; q++) {
            order[at + q] = g;
            opart[at + q] = (uint8_t)q;
        }
    }
}

// MAC thresholds: the smallest integer D with fl(theta^2 * D) > s^2 (FP64,
// theta^2 = theta * theta rounded once), so that "d^2 >= thr" is exactly the
// FP64 test s^2 < theta^2 d^2 on integer grid distances.
MacTable mac_table(float theta) {
    MacTable t;
    double th2 = (double)theta * (double)theta;
    for (int l = 0; l < kLevels; l++) {
        double s2 = ldexp(1.0, 2 * (kMaxLevel - l));
        if (!(th2 > 0.0)) { t.thr[l] = ~0ull; continue; }
        unsigned long long lo = 0, hi = 1ull << 53;
        if (!(th2 * (double)hi > s2)) { t.thr[l] = ~0ull; continue; }  // no grid distance can pass
        while (lo < hi) {
            unsigned long long mid = lo + (hi - lo) / 2;
            if (th2 * (double)mid > s2) hi = mid; else lo = mid + 1;
        }
        t.thr[l] = lo;
    }
    return t;
}

template <bool SOFT, bool QUAD, bool REC, bool REL = false, bool SPL = false>
static cudaError_t launch_walk(rv_ctx *c, const WalkArgs &A, cudaStream_t s) {
    const size_t smem = warp_smem_bytes(A.tile) * kWalkWarps;
    auto kern = walk_tree_k<SOFT, QUAD, REC, REL, SPL>;
    // resident blocks, asked once per context and variant (the tile is the context's). The
    // attribute is the function's, shared by all contexts: always the largest tile's need.
    int &blocks = c->walk_blocks[(REL ? 8 : 0) + (REC ? 4 : (SPL ? 4 : 0) + (SOFT ? 2 : 0) + (QUAD ? 1 : 0))];
    if (blocks == 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)warp_smem_bytes(256) * kWalkWarps);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWalkWarps * 32, smem);
        if (e != cudaSuccess) return e;
        // every warp of the launch has its stack spill area
        blocks = std::min(std::max(1, per_sm) * c->num_sms, kStackSpillWarps / kWalkWarps);
    }
    // no more warps than work items: at most one a star
    const int64_t items = c->n + A.n_extra;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(blocks, (items + kWalkWarps - 1) / kWalkWarps));
    kern<<<grid, kWalkWarps * 32, smem, s>>>(A);
    count_launch(c);
    return cudaGetLastError();
}

rv_status tree_walk(rv_ctx *c, float theta, float eps_star, int n_extra, const float *xyzm, const float *xeps,
                    const int *xmem, int extras_per_member, float *ax, float *ay, float *az, float *pot,
                    float *xout, cudaStream_t s, const PairRecord *rec, const RelMac *rel, const uint8_t *gact,
                    const float4 *xquad, const uint8_t *xq_skip) {
    Workspace &w = c->w;
    WalkArgs A;
    A.pos = w.pos;
    A.cbox = w.cbox;
    A.clink = reinterpret_cast<const int4 *>(w.clink);
    A.cmom = w.cmom;
    A.groups = w.groups;
    A.perm = w.perm;
    A.st = w.st;
    A.cell_cap = (int)c->cell_cap;
    A.n = (int)c->n;
    A.moff = w.moff;
    A.M = c->n_members;
    A.mbounds = w.mbounds;
    A.mroot = w.mroot;
    A.xmem = xmem;
    A.extra_per_member = extras_per_member;
    A.mac = mac_table(theta);
    A.eps2 = eps_star * eps_star;
    A.eps_star = eps_star;
    A.tile = c->cfg.tile;
    A.n_extra = n_extra;
    A.xyzm = xyzm;
    A.xeps = xeps;
    A.xquad = n_extra > 0 ? xquad : nullptr;
    A.xq_skip = xq_skip;
    A.ax = ax; A.ay = ay; A.az = az; A.pot = pot;
    A.xout = xout;
    A.pairs = rec ? rec->pairs : nullptr;
    A.npairs = rec ? rec->npairs : nullptr;
    A.pair_cap = rec ? rec->cap : 0;
    if (rec) A.rec = mac_table(rec->theta_rec);
    A.gact = gact;
    A.gstack = w.gstack;
    A.order = c->n >= kOrderMinStars ? w.gorder : nullptr;
    A.opart = w.gopart;
    A.scost = w.scost;
    A.n_leaf = c->cfg.n_leaf;
    A.parts = parts_of(c->n, c->n_members, c->cfg.group);
    A.partial = w.gpartial;
    A.garrive = w.garrive;
    const bool spline = c->cfg.softening == 1 && eps_star > 0.f;
    {
        const float h = 2.8f * eps_star;
        A.spl.h2 = h * h;
        A.spl.hinv = spline ? 1.f / h : 0.f;
        A.spl.hinv3 = A.spl.hinv * A.spl.hinv * A.spl.hinv;
    }
    A.rel_alpha = rel ? rel->alpha : 0.f;
    A.arx = rel ? rel->rx : nullptr;
    A.ary = rel ? rel->ry : nullptr;
    A.arz = rel ? rel->rz : nullptr;
    if (rel && rec) return set_err(c, RV_E_INVAL, "no pair record under the relative criterion");
    // reset the work counter and statistics
    cudaError_t e = cudaMemsetAsync(&w.st->walk, 0, sizeof(w.st->walk), s);
    if (e != cudaSuccess) return cuda_check(c, e, "walk reset");
    if (c->n == 0 && n_extra == 0) return RV_OK;
    const bool quad = c->cfg.quadrupole != 0;
    // optional timing of this launch on its own stream (not while a graph is being captured)
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (c->profile_walk) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(s, &cs);
        if (cs == cudaStreamCaptureStatusNone) {
            if (c->n_walk_events == c->cap_walk_events) {
                int cap = c->cap_walk_events ? 2 * c->cap_walk_events : 64;
                cudaEvent_t *ev = (cudaEvent_t *)realloc(c->walk_events, sizeof(cudaEvent_t) * 2 * cap);
                if (!ev) return set_err(c, RV_E_CUDA, "walk timing events");
                for (int k = 2 * c->cap_walk_events; k < 2 * cap; k++) ev[k] = nullptr;
                c->walk_events = ev;
                c->cap_walk_events = cap;
            }
            cudaEvent_t *pair = c->walk_events + 2 * c->n_walk_events;
            if (!pair[0]) cudaEventCreate(&pair[0]);
            if (!pair[1]) cudaEventCreate(&pair[1]);
            ev0 = pair[0];
            ev1 = pair[1];
            c->n_walk_events++;
        }
    }
    if (ev0) cudaEventRecord(ev0, s);
    if (A.order) {
        int *bins = w.obins, *gbin = w.gbin;
        const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((c->n + 255) / 256, (int64_t)c->num_sms * 4));
        e = cudaMemsetAsync(bins, 0, sizeof(int) * kOrderBins, s);
        if (e != cudaSuccess) return cuda_check(c, e, "walk order");
        group_bins_k<<<grid, 256, 0, s>>>(OrderArgs{w.groups, w.perm, w.scost, A.parts, (int)c->n}, w.st, gbin, bins);
        group_bins_scan_k<<<1, kOrderBins, 0, s>>>(w.st, (int)c->n, bins);
        group_scatter_k<<<grid, 256, 0, s>>>(w.st, gbin, bins, w.gorder, w.gopart);
        c->launches += 3;
    }
    if (spline) {
        if (rec) return set_err(c, RV_E_INVAL, "no pair record with spline softening");
        if (rel)
            e = quad ? launch_walk<true, true, false, true, true>(c, A, s)
                     : launch_walk<true, false, false, true, true>(c, A, s);
        else
            e = quad ? launch_walk<true, true, false, false, true>(c, A, s)
                     : launch_walk<true, false, false, false, true>(c, A, s);
    } else if (rel) {
        if (eps_star > 0.f)
            e = quad ? launch_walk<true, true, false, true>(c, A, s) : launch_walk<true, false, false, true>(c, A, s);
        else
            e = quad ? launch_walk<false, true, false, true>(c, A, s) : launch_walk<false, false, false, true>(c, A, s);
    } else if (rec) {
        if (!(eps_star > 0.f) || !quad) return set_err(c, RV_E_INVAL, "pair record needs softening and quadrupoles");
        e = launch_walk<true, true, true>(c, A, s);
    } else if (eps_star > 0.f) {
        e = quad ? launch_walk<true, true, false>(c, A, s) : launch_walk<true, false, false>(c, A, s);
    } else {
        e = quad ? launch_walk<false, true, false>(c, A, s) : launch_walk<false, false, false>(c, A, s);
    }
    if (ev1) cudaEventRecord(ev1, s);
    if (e != cudaSuccess) return cuda_check(c, e, "walk launch");
    return RV_OK;
}

}  // namespace rv

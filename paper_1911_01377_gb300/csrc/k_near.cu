/*
 * k_near.cu -- near part of the u-series, Eq. 20:
 *   N(r) = 1/r - F(r) for r < r_c, 0 otherwise
 *   phi_i^near = sum_j q_j N(r_ij),   F_i^near = q_i sum_j q_j (1/r^3 + F'(r)/r) (r_i - r_j)
 * over all j != i and periodic images.
 *
 * Half-list cluster-pair kernel (k_near_half).  Each cell's atoms come in
 * 8-atom spatial clusters (k_cluster_build), and the clusters of a cell in groups
 * of GI consecutive clusters.  One warp owns one group and walks the j-clusters
 * of its own cell (from the group's first cluster on) and of the 13 neighbour
 * cells whose offset (dz, dy, dx) is lexicographically positive, so that every
 * unordered pair and periodic image is visited exactly once (cells have edge
 * >= r_c and there are >= 3 per axis, so the 27 offsets are distinct images).
 * For 32 candidate j-clusters at a time, each lane tests one candidate's
 * bounding box against the GI i-cluster boxes (a conservative test with the
 * pair distance's rounding); a surviving j-cluster is then evaluated against
 * every i-cluster of the group it reaches, one 8 x 8 step each.
 *
 * Lane layout of a step: lane = (jl = lane % 8, gi = lane / 8) holds j atom jl
 * and the i atoms gi and gi + 4 as a two-wide FP32 pair (add/sub/mul/fma.f32x2),
 * so a step covers all 64 pairs of a cluster pair.  i-side sums stay in
 * registers for the whole walk; j-side sums stay in registers while one
 * j-cluster meets the group's i-clusters, are then reduce-scattered over the
 * four lanes of each j atom (lane gi ends with component gi), and added to the
 * atom's accumulator.  Accumulators are 64-bit integers in fixed point (2^-32):
 * integer addition is associative, so the result is the same bits whatever the
 * order in which warps add their parts (deterministic, no floating-point
 * atomics), and the sum is exact.  Each part is an FP32 sum formed in a fixed
 * order, rounded once to the fixed-point grid.
 *
 * The i atoms of a group, its boxes and a unit's neighbour cells lie in the warp's shared memory; the unit's
 * candidates (all its cells together) are tested 32 at a time, the next surviving j-cluster's atoms are loaded
 * while the current one's steps run, and the next unit is taken from the queue during the current one.
 *
 * Bound: issue slots and the latency of the step's chain (57 to 61 % of the slots used at 16 warps per SM; FMA pipe
 * 20 to 23 %, L1 28 to 33 %).  Alone, slab at r_c = 8 / 10 / 13 A:
 * 76 / 98 / 179 us, 200 k charges at 9 A 246 us, 1.06 M at 10 A 1.44 ms, against 92 / 126 / 212 us, 305 us and 1.75
 * ms with i atoms in registers, clusters in Morton order and one scan per neighbour cell.  Not kept: constants
 * pinned in registers (no change: the instructions take them from constant memory); the surviving clusters as a
 * list in shared memory (the loop is no longer uniform: 110 us at 10 A); 3, 5, 6, 7 or 8 CTAs per SM.
 *
 * Per pair: r^2 by the single-precision predicate on d = x_i - (x_j + shift);
 * 1/r by rsqrt; F(u = r^2) = explicit narrow Gaussians plus a polynomial in
 * s = 2u / r_c^2 - 1 (Horner, value and derivative).
 *
 * k_pairs_count is the full-list form used only to list pairs: every directed
 * pair (i, j) with the predicate evaluated from i's side, partner counts and
 * index hashes per atom (the canonical list the oracle reproduces bit for bit).
 */
#include <algorithm>

#include "usr_internal.h"

#ifndef USR_NEAR_GI
#define USR_NEAR_GI 4
#endif
#ifndef USR_NEAR_MINB
#define USR_NEAR_MINB 5     // CTAs of 128 threads per SM the register budget is set for (90 registers used; 4
                            // CTAs then leave 16 k registers of an SM to the far chain)
#endif

namespace usr {

__device__ __forceinline__ unsigned long long mix64(unsigned long long x)
{
    unsigned long long z = x + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

/*
 * Two-wide FP32 arithmetic (the add/mul/fma .f32x2 instructions through
 * CUDA's float2 builtins): each lane evaluates its two pairs of a cluster
 * pair in one instruction stream, halving the issued instructions of the
 * pair arithmetic.  Each element is rounded exactly as the scalar instruction
 * would round it (a - b is formed as a + (-b), which is the same number).
 */
typedef float2 f2;

__device__ __forceinline__ f2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float exp2_ftz(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

/* ------------------------------------------------------------ half list */

constexpr float kFixScale = 4294967296.0f;   // 2^32 fixed-point units per unit of force or potential
constexpr float kFixMax = 1073741824.0f;     // 2^30: largest magnitude one part may carry

/* Add v to a fixed-point accumulator (status bit 8 for a part out of range or NaN). */
__device__ __forceinline__ void red_fix(unsigned long long* p, float v, int* status)
{
    if (!(fabsf(v) < kFixMax)) {
        atomicOr(status, 8);
        return;
    }
    atomicAdd(p, (unsigned long long)__float2ll_rn(v * kFixScale));   // two's complement: a signed add
}

struct NearVir {
    f2 xx, yy, zz, xy, xz, yz;
};

/* i-side sums of one i-cluster, seen by a lane: atoms gi and gi + 4. */
struct NearSum {
    f2 x, y, z, p;
};

/*
 * One 8 x 8 step between the i atoms in A = (x, x', y, y'), B = (z, z', q, q') (atoms gi and gi + 4 of an
 * i-cluster) and the lane's j atom (xj/yj/zj: minus its position shifted to the image, duplicated into both
 * halves).  Padding rows never pass the distance test: as j atoms they sit near -1e6 (cpos), as i atoms near
 * +1e7 (replaced when the group is loaded).  TRI: the j-cluster is the i-cluster itself, only pairs with j
 * after i count (tri_a / tri_b for halves a / b).
 */
template <int DEG, int NEXP, bool VIR, bool TRI>
__device__ __forceinline__ void pair_step(const NearArgs& a, float4 A, float4 B, NearSum& I, f2 xj, f2 yj, f2 zj,
                                          float qj, bool tri_a, bool tri_b, NearSum& J, NearVir& V)
{
    const f2 dx = add2(pk(A.x, A.y), xj), dy = add2(pk(A.z, A.w), yj), dz = add2(pk(B.x, B.y), zj);
    const f2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
    bool ina = r2.x < a.rc2, inb = r2.y < a.rc2;
    if (TRI) {
        ina = ina && tri_a;
        inb = inb && tri_b;
    }
    if (!__any_sync(0xffffffffu, ina || inb)) return;
    // pairs outside r_c (or not counted) get r^2 = r_c^2 and charge 0 on both sides: finite, adds 0
    const float ua = ina ? r2.x : a.rc2, ub = inb ? r2.y : a.rc2;
    const f2 u = pk(ua, ub);
    const f2 ri = pk(rsqrt_ftz(ua), rsqrt_ftz(ub));
    // pn = -F(u), d2 = 2 dF/du: two Horner chains side by side, so that N = 1/r + pn needs no sign change
    const f2 s = fma2(u, a.sfac, dup(-1.0f));
    f2 pn = a.npoly[DEG], d2 = a.dpoly[DEG - 1];
    #pragma unroll
    for (int d = DEG - 1; d >= 0; --d) {
        pn = fma2(pn, s, a.npoly[d]);
        if (d > 0) d2 = fma2(d2, s, a.dpoly[d - 1]);
    }
    const int nexp = NEXP >= 0 ? NEXP : a.n_explicit;
    #pragma unroll
    for (int e = 0; e < nexp; ++e) {
        const f2 t = mul2(u, a.el2[e]);
        const f2 x = pk(exp2_ftz(t.x), exp2_ftz(t.y));
        pn = fma2(x, a.nea[e], pn);
        d2 = fma2(x, a.dea[e], d2);
    }
    const f2 nr = add2(ri, pn);                                           // N(r) = 1/r - F
    const f2 g = fma2(mul2(ri, ri), ri, d2);                              // -N'(r) / r
    const f2 Qj = pk(ina ? qj : 0.f, inb ? qj : 0.f);
    const f2 Qi = pk(ina ? B.z : 0.f, inb ? B.w : 0.f);
    const f2 gi = mul2(g, Qj);
    I.x = fma2(gi, dx, I.x);
    I.y = fma2(gi, dy, I.y);
    I.z = fma2(gi, dz, I.z);
    I.p = fma2(nr, Qj, I.p);
    const f2 gj = mul2(g, Qi);
    J.x = fma2(gj, dx, J.x);
    J.y = fma2(gj, dy, J.y);
    J.z = fma2(gj, dz, J.z);
    J.p = fma2(nr, Qi, J.p);
    if (VIR) {
        // q_i q_j g d (x) d over the pairs (each unordered pair once)
        const f2 w = mul2(gi, pk(B.z, B.w));
        const f2 wx = mul2(w, dx), wy = mul2(w, dy);
        V.xx = fma2(wx, dx, V.xx);
        V.xy = fma2(wx, dy, V.xy);
        V.xz = fma2(wx, dz, V.xz);
        V.yy = fma2(wy, dy, V.yy);
        V.yz = fma2(wy, dz, V.yz);
        V.zz = fma2(mul2(w, dz), dz, V.zz);
    }
}

/*
 * The half-shell neighbour cells of a work unit: offsets nb = 13 (the own cell) .. 26 split into kNearSplits
 * ranges of kSplitCells cells.
 */
constexpr int kNearSplits = 7, kSplitCells = (14 + kNearSplits - 1) / kNearSplits;

/* A warp's shared memory: its group's i atoms in the paired layout (per cluster four 32-byte rows gi: x, x', y,
   y', z, z', q, q' of atoms gi and gi + 4), their boxes, and the unit's neighbour cells: candidate t of cell k
   (end[k - 1] <= t < end[k]) is cluster off[k] + t, at image shift sh[k]. */
template <int GI>
struct NearShared {
    float4 ipos[GI][8];
    float4 box[GI][2];
    float4 sh[kSplitCells];
    int off[kSplitCells], end[kSplitCells];
};

/* The group of work unit u into d (a warp's next unit); units when there is none. */
__device__ __forceinline__ int near_next(const ClusterList& L, const NearArgs& a, int u, int units, int4& d,
                                         int* __restrict__ status)
{
    if (u >= units || !USR_IN_BOUNDS(u / kNearSplits, a.max_groups, status)) return units;
    d = L.gdesc[u / kNearSplits];
    return u;
}

/*
 * One work unit: group d = (first cluster, cell, clusters) (its GI clusters' i atoms) against the j-clusters of
 * the neighbour offsets nb0 .. nb1 - 1.  Adds the i- and j-side parts to acc; VIR: writes the unit's pair virial
 * sum_pairs d (x) f (six FP64 values) to vir.  Takes the warp's next unit from the queue on the way (`next`) and
 * loads its group into dn, so that those two dependent reads are not waited for.
 */
template <int GI, int DEG, int NEXP, bool VIR>
__device__ __forceinline__ void near_unit(const ClusterList& L, const NearArgs& a, int4 d, int nb0, int nb1,
                                          NearShared<GI>& S, unsigned long long* __restrict__ acc,
                                          double* __restrict__ vir, int* __restrict__ queue, int units, int& next,
                                          int4& dn, int* __restrict__ status)
{
    static_assert(GI * 8 == 32, "one lane per i atom of the group");
    const int lane = threadIdx.x & 31;
    const int ncx = a.box.nc[0], ncy = a.box.nc[1], ncz = a.box.nc[2];
    const int c0 = d.x, cell = d.y, ni = d.z;
    int ticket = 0;
    if (lane == 0) ticket = atomicAdd(queue, 1);
    const int jl = lane & 7, gi = lane >> 3;
    const int ncells = nb1 - nb0;
    {
        // the group's atoms, one per lane; padding rows (near -1e6) move to +1e7, far from every j position
        float4 p = make_float4(1.0e7f, 1.0e7f, 1.0e7f, 0.f);
        if (gi < ni) p = L.cpos[c0 * 8 + lane];
        if (p.x < -5.0e5f) p = make_float4(1.0e7f, 1.0e7f, 1.0e7f, 0.f);
        float* row = reinterpret_cast<float*>(&S.ipos[gi][2 * (jl & 3)]) + (jl >> 2);
        row[0] = p.x;
        row[2] = p.y;
        row[4] = p.z;
        row[6] = p.w;
    }
    if (lane < 2 * GI) {
        const int k = lane >> 1;
        float4 v;
        if (k < ni) v = (lane & 1) ? L.bbhi[c0 + k] : L.bblo[c0 + k];
        else v = (lane & 1) ? make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f) : make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f);
        S.box[k][lane & 1] = v;
    }
    int total;
    {
        // lane k < ncells: neighbour cell nb0 + k, its image shift and cluster range
        const int cx = cell % ncx, cy = (cell / ncx) % ncy, cz = cell / (ncx * ncy);
        const int nb = nb0 + min(lane, ncells - 1);
        int nx = cx + nb % 3 - 1, ny = cy + (nb / 3) % 3 - 1, nz = cz + nb / 9 - 1;
        float sx = 0.f, sy = 0.f, sz = 0.f;
        if (nx < 0) { nx += ncx; sx = -a.box.L[0]; } else if (nx >= ncx) { nx -= ncx; sx = a.box.L[0]; }
        if (ny < 0) { ny += ncy; sy = -a.box.L[1]; } else if (ny >= ncy) { ny -= ncy; sy = a.box.L[1]; }
        if (nz < 0) { nz += ncz; sz = -a.box.L[2]; } else if (nz >= ncz) { nz -= ncz; sz = a.box.L[2]; }
        const int nc = (nz * ncy + ny) * ncx + nx;
        const int jc0 = nb == 13 ? c0 : L.pstart[nc] >> 3, jc1 = L.pstart[nc + 1] >> 3;
        const int cnt = lane < ncells ? jc1 - jc0 : 0;
        int inc = cnt;
        #pragma unroll
        for (int o = 1; o < kSplitCells; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        total = __shfl_sync(0xffffffffu, inc, kSplitCells - 1);
        if (lane < kSplitCells) {
            S.sh[lane] = make_float4(sx, sy, sz, 0.f);
            S.off[lane] = jc0 - (inc - cnt);
            S.end[lane] = inc;
        }
    }
    __syncwarp();
    NearSum I[GI];
    #pragma unroll
    for (int k = 0; k < GI; ++k) I[k].x = I[k].y = I[k].z = I[k].p = dup(0.f);
    NearVir V;
    V.xx = V.yy = V.zz = V.xy = V.xz = V.yz = dup(0.f);
    const bool tri_a = jl > gi, tri_b = jl > gi + 4;
    const bool b1 = (lane & 16) != 0, b0 = (lane & 8) != 0;
    if (total == 0) next = near_next(L, a, __shfl_sync(0xffffffffu, ticket, 0), units, dn, status);
    // clusters of the unit's own cell come first: candidate t < GI is cluster c0 + t, one of the group's own
    const int nown = nb0 == 13 ? ni : 0;
    int ends[kSplitCells];                 // uniform copies
    #pragma unroll
    for (int k = 0; k < kSplitCells; ++k) ends[k] = S.end[k];
    auto cell_of = [&](int t) {
        int k = 0;
        #pragma unroll
        for (int c = 0; c + 1 < kSplitCells; ++c) k += t >= ends[c];
        return k;
    };
    for (int tb = 0; tb < total; tb += 32) {
        unsigned int m = 0;
        {
            const int t = tb + lane;
            const int k = cell_of(t);
            if (t < total) {
                const int jc = S.off[k] + t;
                if (USR_IN_BOUNDS(jc, a.max_clusters, status)) {
                    const float4 lo = L.bblo[jc], hi = L.bbhi[jc], sh = S.sh[k];
                    const float lx = __fadd_rn(lo.x, sh.x), ly = __fadd_rn(lo.y, sh.y), lz = __fadd_rn(lo.z, sh.z);
                    const float hx = __fadd_rn(hi.x, sh.x), hy = __fadd_rn(hi.y, sh.y), hz = __fadd_rn(hi.z, sh.z);
                    #pragma unroll
                    for (int i = 0; i < GI; ++i) {
                        const float4 blo = S.box[i][0], bhi = S.box[i][1];
                        // gap between the boxes, rounded like a pair distance
                        const float gx = fmaxf(0.f, fmaxf(__fsub_rn(lx, bhi.x), __fsub_rn(blo.x, hx)));
                        const float gy = fmaxf(0.f, fmaxf(__fsub_rn(ly, bhi.y), __fsub_rn(blo.y, hy)));
                        const float gz = fmaxf(0.f, fmaxf(__fsub_rn(lz, bhi.z), __fsub_rn(blo.z, hz)));
                        if (__fmaf_rn(gz, gz, __fmaf_rn(gy, gy, __fmul_rn(gx, gx))) < a.rc2) m |= 1u << i;
                    }
                    // own cell: i-cluster c0 + k meets j-clusters from c0 + k on
                    if (t < nown) m &= (2u << t) - 1u;
                }
            }
        }
        if (tb == 0) next = near_next(L, a, __shfl_sync(0xffffffffu, ticket, 0), units, dn, status);
        unsigned int bal = __ballot_sync(0xffffffffu, m != 0);
        if (!bal) continue;
        // the surviving j-clusters; the next one's atoms are loaded while this one's steps run
        int t = __ffs(bal) - 1;
        int tc = tb + t;
        int k = cell_of(tc);
        int jcl = S.off[k] + tc;
        float4 pj = L.cpos[jcl * 8 + jl];
        for (;;) {
            bal &= bal - 1;
            const float4 sh = S.sh[k];
            const unsigned int mk = __shfl_sync(0xffffffffu, m, t);
            const int jcur = jcl;
            const bool own = tc < nown;
            // minus the image position, -(x_j + shift): d = x_i + that, the same number as x_i - (x_j + shift)
            const f2 xj = dup(-__fadd_rn(pj.x, sh.x)), yj = dup(-__fadd_rn(pj.y, sh.y)), zj = dup(-__fadd_rn(pj.z, sh.z));
            const float qj = pj.w;
            const int own_k = tc;
            if (bal) {
                t = __ffs(bal) - 1;
                tc = tb + t;
                k = cell_of(tc);
                jcl = S.off[k] + tc;
                pj = L.cpos[jcl * 8 + jl];
            }
            NearSum J;
            J.x = J.y = J.z = J.p = dup(0.f);
            if (own) {
                // the j-cluster is one of the group's own: that step counts j after i only
                #pragma unroll
                for (int i = 0; i < GI; ++i)
                    if (mk & (1u << i)) {
                        const float4 A = S.ipos[i][2 * gi], B = S.ipos[i][2 * gi + 1];
                        if (own_k == i)
                            pair_step<DEG, NEXP, VIR, true>(a, A, B, I[i], xj, yj, zj, qj, tri_a, tri_b, J, V);
                        else
                            pair_step<DEG, NEXP, VIR, false>(a, A, B, I[i], xj, yj, zj, qj, tri_a, tri_b, J, V);
                    }
            } else {
                #pragma unroll
                for (int i = 0; i < GI; ++i)
                    if (mk & (1u << i)) {
                        const float4 A = S.ipos[i][2 * gi], B = S.ipos[i][2 * gi + 1];
                        pair_step<DEG, NEXP, VIR, false>(a, A, B, I[i], xj, yj, zj, qj, tri_a, tri_b, J, V);
                    }
            }
            // j-side sums: fold the two i halves, reduce-scatter over the four lanes gi of atom jl; lane
            // (jl, gi) ends with component gi, which is accumulator `lane` of the cluster
            const float vx = J.x.x + J.x.y, vy = J.y.x + J.y.y;
            const float vz = J.z.x + J.z.y, vp = J.p.x + J.p.y;
            const float r0 = __shfl_xor_sync(0xffffffffu, b1 ? vx : vz, 16);
            const float r1 = __shfl_xor_sync(0xffffffffu, b1 ? vy : vp, 16);
            const float k0 = (b1 ? vz : vx) + r0, k1 = (b1 ? vp : vy) + r1;
            const float r2 = __shfl_xor_sync(0xffffffffu, b0 ? k0 : k1, 8);
            const float v = (b0 ? k1 : k0) + r2;
            if (USR_IN_BOUNDS(jcur, a.max_clusters, status))
                red_fix(acc + 32 * (size_t)jcur + lane, gi < 3 ? -qj * v : v, status);
            if (!bal) break;
        }
    }
    // i-side sums: reduce-scatter the 8 values of each cluster (2 atoms x 4 components) over the 8
    // lanes jl; lane (jl, gi) ends with component jl % 4 of atom gi + 4 (jl / 4)
    const bool c2 = (lane & 4) != 0, c1 = (lane & 2) != 0, c0b = (lane & 1) != 0;
    #pragma unroll
    for (int k = 0; k < GI; ++k) {
        if (k >= ni) break;
        const float va[4] = {I[k].x.x, I[k].y.x, I[k].z.x, I[k].p.x};
        const float vb[4] = {I[k].x.y, I[k].y.y, I[k].z.y, I[k].p.y};
        float w4[4];
        #pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float r = __shfl_xor_sync(0xffffffffu, c2 ? va[m] : vb[m], 4);
            w4[m] = (c2 ? vb[m] : va[m]) + r;
        }
        float w2[2];
        #pragma unroll
        for (int m = 0; m < 2; ++m) {
            const float r = __shfl_xor_sync(0xffffffffu, c1 ? w4[m] : w4[m + 2], 2);
            w2[m] = (c1 ? w4[m + 2] : w4[m]) + r;
        }
        const float r = __shfl_xor_sync(0xffffffffu, c0b ? w2[0] : w2[1], 1);
        const float v = (c0b ? w2[1] : w2[0]) + r;
        const int comp = jl & 3;
        const float4 B = S.ipos[k][2 * gi + 1];
        const float qi = c2 ? B.w : B.z;
        red_fix(acc + 32 * (size_t)(c0 + k) + 8 * comp + gi + 4 * (jl >> 2), comp < 3 ? qi * v : v, status);
    }
    if (VIR) {
        const f2 vv[6] = {V.xx, V.yy, V.zz, V.xy, V.xz, V.yz};
        double v6[6];
        #pragma unroll
        for (int c6 = 0; c6 < 6; ++c6) v6[c6] = (double)(vv[c6].x + vv[c6].y);
        #pragma unroll
        for (int c6 = 0; c6 < 6; ++c6)
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) v6[c6] += __shfl_xor_sync(0xffffffffu, v6[c6], o);
        if (lane == 0)
            for (int c6 = 0; c6 < 6; ++c6) vir[c6] = v6[c6];
    }
    __syncwarp();   // S is rewritten by the warp's next unit
}

/*
 * Persistent warps: each takes work units (group, neighbour range) from a queue counter (zeroed by
 * the cell-list scan), full groups first and the partial ones last, until none is left.  The
 * accumulation is integer, so results do not depend on which warp takes which unit.  acc: 4
 * fixed-point accumulators (Fx, Fy, Fz, phi) per cluster slot, zeroed by k_cluster_build.  VIR: unit u
 * writes its pair virial to vir[6 u ..].
 */
template <int GI, int DEG, int NEXP, bool VIR>
__global__ void __launch_bounds__(128, USR_NEAR_MINB) k_near_half(ClusterList L, const __grid_constant__ NearArgs a,
                                                                    int* __restrict__ queue,
                                                                    unsigned long long* __restrict__ acc,
                                                                    double* __restrict__ vir, int* __restrict__ status)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    __shared__ NearShared<GI> S[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ncell = a.box.nc[0] * a.box.nc[1] * a.box.nc[2];
    const int units = kNearSplits * (L.gfull[ncell] + L.gpart[ncell]);
    int u = 0;
    if (lane == 0) u = atomicAdd(queue, 1);
    int4 d = make_int4(0, 0, 0, 0);
    u = near_next(L, a, __shfl_sync(0xffffffffu, u, 0), units, d, status);
    while (u < units) {
        const int sub = u % kNearSplits, nb0 = 13 + sub * kSplitCells, nb1 = min(27, nb0 + kSplitCells);
        if (!USR_IN_BOUNDS(d.x + d.z - 1, a.max_clusters, status)) return;
        int next = units;
        int4 dn = d;
        near_unit<GI, DEG, NEXP, VIR>(L, a, d, nb0, nb1, S[warp], acc, VIR ? vir + 6 * (size_t)u : nullptr, queue,
                                      units, next, dn, status);
        u = next;
        d = dn;
    }
}

/* ------------------------------------------------------------ pair listing */

/*
 * Full list, one warp per i-cluster, lane (il = lane / 4, g = lane % 4) with
 * i atom il and j atoms g and g + 4: partners j != i with r^2 < r_c^2 under the
 * single-precision predicate d = x_i - (x_j + shift), evaluated from i's side;
 * count and the sum of splitmix64 of the partners' caller indices.
 */
__global__ void __launch_bounds__(128) k_pairs_count(ClusterList L, NearArgs a,
                                                     int* __restrict__ count, unsigned long long* __restrict__ hash,
                                                     int* __restrict__ status)
{
    const int ncx = a.box.nc[0], ncy = a.box.nc[1], ncz = a.box.nc[2];
    const int ncl = L.pstart[ncx * ncy * ncz] >> 3;
    const int ic = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (ic >= ncl || !USR_IN_BOUNDS(ic, a.max_clusters, status)) return;
    const int il = lane >> 2, g = lane & 3;
    const int islot = ic * 8 + il;
    const float4 pi = L.cpos[islot];
    const f2 pix = dup(pi.x), piy = dup(pi.y), piz = dup(pi.z);
    const float4 blo = L.bblo[ic], bhi = L.bbhi[ic];
    const int c = L.ccell[ic];
    const int cx = c % ncx, cy = (c / ncx) % ncy, cz = c / (ncx * ncy);
    int cnt = 0;
    unsigned long long h = 0ull;
    for (int nb = 0; nb < 27; ++nb) {
        int nx = cx + nb % 3 - 1, ny = cy + (nb / 3) % 3 - 1, nz = cz + nb / 9 - 1;
        float sx = 0.f, sy = 0.f, sz = 0.f;
        if (nx < 0) { nx += ncx; sx = -a.box.L[0]; } else if (nx >= ncx) { nx -= ncx; sx = a.box.L[0]; }
        if (ny < 0) { ny += ncy; sy = -a.box.L[1]; } else if (ny >= ncy) { ny -= ncy; sy = a.box.L[1]; }
        if (nz < 0) { nz += ncz; sz = -a.box.L[2]; } else if (nz >= ncz) { nz -= ncz; sz = a.box.L[2]; }
        const f2 sx2 = dup(sx), sy2 = dup(sy), sz2 = dup(sz);
        const int nc = (nz * ncy + ny) * ncx + nx;
        const int jc0 = L.pstart[nc] >> 3, jc1 = L.pstart[nc + 1] >> 3;
        for (int jb = jc0; jb < jc1; jb += 32) {
            const int jc = jb + lane;
            bool near = false;
            if (jc < jc1 && USR_IN_BOUNDS(jc, a.max_clusters, status)) {
                const float4 lo = L.bblo[jc], hi = L.bbhi[jc];
                const float gx = fmaxf(0.f, fmaxf(__fsub_rn(__fadd_rn(lo.x, sx), bhi.x), __fsub_rn(blo.x, __fadd_rn(hi.x, sx))));
                const float gy = fmaxf(0.f, fmaxf(__fsub_rn(__fadd_rn(lo.y, sy), bhi.y), __fsub_rn(blo.y, __fadd_rn(hi.y, sy))));
                const float gz = fmaxf(0.f, fmaxf(__fsub_rn(__fadd_rn(lo.z, sz), bhi.z), __fsub_rn(blo.z, __fadd_rn(hi.z, sz))));
                near = __fmaf_rn(gz, gz, __fmaf_rn(gy, gy, __fmul_rn(gx, gx))) < a.rc2;
            }
            unsigned int m = __ballot_sync(0xffffffffu, near);
            while (m) {
                const int k = __ffs(m) - 1;
                m &= m - 1;
                const int jcl = jb + k;
                const float4 A = L.cpos[jcl * 8 + g], B = L.cpos[jcl * 8 + 4 + g];
                const f2 dx = sub2(pix, add2(pk(A.x, B.x), sx2));
                const f2 dy = sub2(piy, add2(pk(A.y, B.y), sy2));
                const f2 dz = sub2(piz, add2(pk(A.z, B.z), sz2));
                const f2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
                const float r2a = r2.x, r2b = r2.y;
                const bool self = nb == 13 && jcl == ic;
                if (r2a < a.rc2 && !(self && g == il)) {
                    ++cnt;
                    h += mix64((unsigned long long)L.cperm[jcl * 8 + g]);
                }
                if (r2b < a.rc2 && !(self && g + 4 == il)) {
                    ++cnt;
                    h += mix64((unsigned long long)L.cperm[jcl * 8 + 4 + g]);
                }
            }
        }
    }
    #pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        h += __shfl_xor_sync(0xffffffffu, h, o);
    }
    const int ci = L.cperm[islot];
    if (g == 0 && ci >= 0) {
        if (USR_IN_BOUNDS(ci, a.max_atoms, status)) {
            count[ci] = cnt;
            hash[ci] = h;
        }
    }
}

/* ------------------------------------------------------------ launchers */

constexpr int kNearGroup = USR_NEAR_GI;

int near_max_groups(int n, int ncell) { return (int)(((long long)n + (8LL * kNearGroup - 1) * ncell) / (8 * kNearGroup)) + 1; }

int near_group_clusters() { return kNearGroup; }

int near_units(int max_groups) { return kNearSplits * max_groups; }

int near_splits() { return kNearSplits; }

/*
 * CTAs per SM the pair kernel's instance can hold, and the SM count (once per instance; thread-safe
 * static initialisation).
 */
template <typename K>
static int2 persistent_shape(K kernel)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 128, 0);
    return make_int2(per_sm > 0 ? per_sm : 1, sms > 0 ? sms : 1);
}

/*
 * Grid of the persistent pair kernel: the CTAs the SMs hold at once, or at most ctas_per_sm per SM when that
 * is given (an evaluation leaves one slot per SM to the far chain beside it); at least one per SM.
 */
static int persistent_grid(int2 shape, int ctas_per_sm, int units_max)
{
    int per_sm = shape.x;
    if (ctas_per_sm > 0) per_sm = std::min(per_sm, ctas_per_sm);
    if (per_sm < 1) per_sm = 1;
    return std::max(1, std::min(per_sm * shape.y, (units_max + 3) / 4));
}

template <int GI, int DEG, int NEXP>
static void launch_half(int max_groups, const ClusterList& L, const NearArgs& a, int* queue, unsigned long long* acc,
                        double* vir, int* status, int ctas_per_sm, cudaStream_t st)
{
    const int units_max = kNearSplits * max_groups;
    if (vir) {
        static const int2 shape = persistent_shape(k_near_half<GI, DEG, NEXP, true>);
        launch_pdl(k_near_half<GI, DEG, NEXP, true>, persistent_grid(shape, ctas_per_sm, units_max), 128, 0, st, L,
                   a, queue, acc, vir, status);
    } else {
        static const int2 shape = persistent_shape(k_near_half<GI, DEG, NEXP, false>);
        launch_pdl(k_near_half<GI, DEG, NEXP, false>, persistent_grid(shape, ctas_per_sm, units_max), 128, 0, st, L,
                   a, queue, acc, nullptr, status);
    }
}

/* One explicit Gaussian (the common case: the narrow j = 0 term) unrolled, any other count in a loop. */
template <int DEG>
static void launch_deg(int max_groups, const ClusterList& L, const NearArgs& a, int* queue, unsigned long long* acc,
                       double* vir, int* status, int ctas_per_sm, cudaStream_t st)
{
    if (a.n_explicit == 1)
        launch_half<kNearGroup, DEG, 1>(max_groups, L, a, queue, acc, vir, status, ctas_per_sm, st);
    else
        launch_half<kNearGroup, DEG, -1>(max_groups, L, a, queue, acc, vir, status, ctas_per_sm, st);
}

void launch_near(int max_groups, int deg, const ClusterList& L, const NearArgs& a, int* queue,
                 unsigned long long* acc, double* vir, int* status, int ctas_per_sm, cudaStream_t st)
{
#define USR_NEAR_DEG(D) \
    case D: launch_deg<D>(max_groups, L, a, queue, acc, vir, status, ctas_per_sm, st); break;
    switch (deg) {
        USR_NEAR_DEG(5)
        USR_NEAR_DEG(6)
        USR_NEAR_DEG(7)
        USR_NEAR_DEG(8)
        USR_NEAR_DEG(10)
        USR_NEAR_DEG(12)
        USR_NEAR_DEG(16)
        USR_NEAR_DEG(20)
        default: launch_deg<24>(max_groups, L, a, queue, acc, vir, status, ctas_per_sm, st); break;
    }
#undef USR_NEAR_DEG
}

void launch_pairs(int max_clusters, const ClusterList& L, const NearArgs& a, int* count,
                  unsigned long long* hash, int* status, cudaStream_t st)
{
    const int blocks = (max_clusters + 3) / 4;
    k_pairs_count<<<blocks, 128, 0, st>>>(L, a, count, hash, status);
}

}  // namespace usr

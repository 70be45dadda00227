/*
 * k_bin.cu -- cell list of the near part (Eq. 20 is range-limited to r_c, so
 * partners of an atom lie in its own or the 26 adjacent cells of edge >= r_c).
 *
 *   bin_count   wrap each position into the box, compute its cell with the
 *               single-precision predicate below, count atoms per cell
 *   scan        exclusive prefix sum of the counts -> cell_start
 *   place       scatter caller indices into their cell's range
 *   cell_sort   order each cell's atoms by caller index (a stable, run-to-run
 *               deterministic order) and gather the sorted float4 rows
 *   clusters    8-atom spatial clusters, the order every later kernel walks (an evaluation does not
 *               run cell_sort)
 *
 * Predicate (per axis, RN rounding, no contraction):
 *   k = floorf(x * invL); xw = fmaf(-k, L, x); if (xw < 0) xw += L;
 *   if (xw >= L) xw -= L; cell = min((int)(xw * cs), nc - 1)
 * Non-finite rows, and rows so far from the box (beyond about 2^22 box
 * lengths) that the wrap leaves them outside [0, L], go to cell 0 at the
 * origin with charge 0 and raise the status word.
 */
#include <climits>

#include "usr_internal.h"

namespace usr {

__device__ __forceinline__ float canon_wrap(float x, float invL, float L)
{
    float k = floorf(__fmul_rn(x, invL));
    float xw = __fmaf_rn(-k, L, x);
    if (xw < 0.0f) xw = __fadd_rn(xw, L);
    if (xw >= L) xw = __fsub_rn(xw, L);
    return xw;
}

__device__ __forceinline__ int canon_cell(float xw, float cs, int nc)
{
    float u = __fmul_rn(xw, cs);
    int c = (u >= 0.0f) ? (int)u : 0;
    return c > nc - 1 ? nc - 1 : c;
}

__global__ void __launch_bounds__(256) k_bin_count(int n, const float4* __restrict__ xyzq, BoxF b,
                                                   int* __restrict__ count, int* __restrict__ cell_of,
                                                   int* __restrict__ slot, float4* __restrict__ wpos,
                                                   ChargeSum* qsum, int* __restrict__ status)
{
    pdl_trigger();   // dependents may be scheduled now; they wait for this grid in pdl_wait
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const unsigned int live = __activemask();
    float4 p = xyzq[i];
    bool ok = isfinite(p.x) && isfinite(p.y) && isfinite(p.z);
    float xw = 0.f, yw = 0.f, zw = 0.f;
    if (ok) {
        xw = canon_wrap(p.x, b.invL[0], b.L[0]);
        yw = canon_wrap(p.y, b.invL[1], b.L[1]);
        zw = canon_wrap(p.z, b.invL[2], b.L[2]);
        // Within 2^22 box lengths of the box the period count floorf(x / L) is off by at most one and the
        // wrapped value lies in [0, L] (L itself only by rounding).  Farther out it can be off by more, and
        // a wrapped value outside the box would send the grid kernels' stencils outside their tiles and
        // grids: such rows are refused like non-finite ones (a zero charge at the origin, status bit 1).
        ok = xw >= 0.0f && xw <= b.L[0] && yw >= 0.0f && yw <= b.L[1] && zw >= 0.0f && zw <= b.L[2];
        if (!ok) xw = yw = zw = 0.0f;
    }
    if (!ok || !isfinite(p.w)) atomicOr(status, 1);
    int cx = canon_cell(xw, b.cs[0], b.nc[0]);
    int cy = canon_cell(yw, b.cs[1], b.nc[1]);
    int cz = canon_cell(zw, b.cs[2], b.nc[2]);
    int c = (cz * b.nc[1] + cy) * b.nc[0] + cx;
    if (!USR_IN_BOUNDS(c, b.nc[0] * b.nc[1] * b.nc[2], status)) c = 0;
    cell_of[i] = c;
    // one atomic per distinct cell in the warp (neighbouring caller indices are often in one cell); the slot
    // order inside a cell is arbitrary either way: k_cluster_build and k_cell_sort order it by keys of their own
    const unsigned int peers = __match_any_sync(live, c);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(&count[c], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    slot[i] = base + __popc(peers & ((1u << lane) - 1u));
    const float q = (ok && isfinite(p.w)) ? p.w : 0.0f;
    wpos[i] = make_float4(xw, yw, zw, q);
    if (qsum) {
        // the largest charge, one atomic per block (a read of the maximum by every warp, to spare most of the atomics,
        // costs 14 us at 1 M charges: all the reads hit one line)
        __shared__ int big[8];
        const int m = __reduce_max_sync(live, __float_as_int(fabsf(q)));
        if (lane == 0) big[threadIdx.x >> 5] = m;
        __syncthreads();         // (threads past n have left)
        if (threadIdx.x == 0) {
            int v = big[0];
            for (int w = 1; 32 * w < min(256, n - (int)(blockIdx.x * 256)); ++w) v = max(v, big[w]);
            atomicMax(&qsum->max_new, v);
        }
    }
}

/*
 * Exclusive scans, one block of 1024 threads: of count[0..ncell) into
 * start[0..ncell] and of the counts rounded up to a multiple of 8 into
 * pstart[0..ncell] (the padded 8-atom cluster layout of the pair kernels).
 * With gfull given, also the half-list pair kernel's groups of gcl
 * consecutive clusters of one cell: the full groups per cell into
 * gfull[0..ncell], the one partial group a cell may end with into
 * gpart[0..ncell]; and the kernel's work-queue counter is set to zero.  With
 * qsum given, the charges' sum is made ready for k_cluster_build.
 */
__global__ void __launch_bounds__(1024) k_scan(int ncell, int* __restrict__ count, int* __restrict__ start,
                                               int* __restrict__ pstart, int* __restrict__ gfull,
                                               int* __restrict__ gpart, int gcl, int* __restrict__ queue,
                                               ChargeSum* __restrict__ qsum)
{
    pdl_trigger();   // dependents may be scheduled now; they wait for this grid in pdl_wait
    pdl_wait();
    __shared__ int4 warp_sums[32];
    __shared__ int4 carry;
    if (threadIdx.x == 0) {
        carry = make_int4(0, 0, 0, 0);
        if (queue) *queue = 0;
        if (qsum) {
            qsum->max = qsum->max_new;
            qsum->max_new = 0;
            qsum->sum = 0ull;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int base = 0; base < ncell; base += 1024) {
        const int i = base + threadIdx.x;
        const int v = i < ncell ? count[i] : 0;
        if (i < ncell) count[i] = 0;   // ready for the next evaluation's counting
        const int vp = (v + 7) & ~7;
        const int vf = (vp >> 3) / gcl, vq = (vp >> 3) % gcl != 0 ? 1 : 0;
        int4 x = make_int4(v, vp, vf, vq);
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int4 y = make_int4(__shfl_up_sync(0xffffffffu, x.x, o), __shfl_up_sync(0xffffffffu, x.y, o),
                                     __shfl_up_sync(0xffffffffu, x.z, o), __shfl_up_sync(0xffffffffu, x.w, o));
            if (lane >= o) { x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w; }
        }
        if (lane == 31) warp_sums[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int4 w = warp_sums[lane];
            #pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int4 y = make_int4(__shfl_up_sync(0xffffffffu, w.x, o), __shfl_up_sync(0xffffffffu, w.y, o),
                                         __shfl_up_sync(0xffffffffu, w.z, o), __shfl_up_sync(0xffffffffu, w.w, o));
                if (lane >= o) { w.x += y.x; w.y += y.y; w.z += y.z; w.w += y.w; }
            }
            warp_sums[lane] = w;   // inclusive
        }
        __syncthreads();
        const int4 pre = wid > 0 ? warp_sums[wid - 1] : make_int4(0, 0, 0, 0);
        const int4 incl = make_int4(x.x + pre.x + carry.x, x.y + pre.y + carry.y, x.z + pre.z + carry.z,
                                    x.w + pre.w + carry.w);
        if (i < ncell) {
            start[i] = incl.x - v;
            pstart[i] = incl.y - vp;
            if (gfull) {
                gfull[i] = incl.z - vf;
                gpart[i] = incl.w - vq;
            }
        }
        __syncthreads();
        if (threadIdx.x == 1023) carry = incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        start[ncell] = carry.x;
        pstart[ncell] = carry.y;
        if (gfull) {
            gfull[ncell] = carry.z;
            gpart[ncell] = carry.w;
        }
    }
}

__global__ void __launch_bounds__(256) k_place(int n, const int* __restrict__ cell_of, const int* __restrict__ slot,
                                               const int* __restrict__ start, int* __restrict__ unsorted,
                                               int* __restrict__ status)
{
    pdl_trigger();   // dependents may be scheduled now; they wait for this grid in pdl_wait
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int d = start[cell_of[i]] + slot[i];
    if (USR_IN_BOUNDS(d, n, status)) unsorted[d] = i;
}

/*
 * One CTA per cell: rank of each entry = number of smaller caller indices in
 * the cell, counted over a shared-memory copy of the cell's entries (all
 * threads read the same element at a time: broadcast, no bank conflicts).
 * Cells larger than the shared copy fall back to counting in global memory.
 */
constexpr int kSortThreads = 128;
constexpr int kSortMax = 2048;

__global__ void __launch_bounds__(kSortThreads) k_cell_sort(int n, const int* __restrict__ start,
                                                            const int* __restrict__ unsorted,
                                                            const float4* __restrict__ wpos, int* __restrict__ perm,
                                                            float4* __restrict__ spos, int* __restrict__ status)
{
    pdl_trigger();   // dependents may be scheduled now; they wait for this grid in pdl_wait
    pdl_wait();
    __shared__ int v[kSortMax];
    const int c = blockIdx.x;
    const int s0 = start[c], m = start[c + 1] - s0;
    if (m == 0) return;
    const bool in_smem = m <= kSortMax;
    if (in_smem)
        for (int e = threadIdx.x; e < m; e += kSortThreads) v[e] = unsorted[s0 + e];
    __syncthreads();
    const int* src = in_smem ? v : unsorted + s0;
    for (int e = threadIdx.x; e < m; e += kSortThreads) {
        const int x = src[e];
        int r = 0;
        for (int f = 0; f < m; ++f) r += src[f] < x;
        if (!USR_IN_BOUNDS(s0 + r, n, status) || !USR_IN_BOUNDS(x, n, status)) continue;
        perm[s0 + r] = x;
        spos[s0 + r] = wpos[x];
    }
}

/*
 * 8-atom clusters for the pair kernel, one CTA per cell.  The cell's atoms are packed by sorting and
 * tiling: sorted by x and cut into slabs, each slab sorted by y and cut into columns, each column sorted
 * by z; every cut falls on a multiple of 8 atoms, so the clusters (runs of 8) are disjoint boxes of about
 * equal edges.  About cbrt(clusters) slabs and the square root of a slab's clusters as columns.  Written to
 * the padded layout at pstart[c] as (x, y, z, q) rows with dummy rows (q = 0, far away and far apart, index
 * -1) after the last atom; then each cluster's bounding box.
 *
 * The pair kernel's work is the 8 x 8 cluster pairs whose boxes come within r_c.  Against runs of 8 along a
 * Morton curve on an 8 x 8 x 8 lattice in the cell (the earlier order, whose runs straddle octants) tiling
 * leaves 20 % fewer of them on the slab at r_c = 10 A and 23 % fewer on water at r_c = 9 A (counted on the
 * CPU), the same as recursive median splits, for three rank-by-counting passes of which the second and third
 * only run over a slab and a column.  The Morton order remains for cells of more than kTileMax atoms, whose
 * three keys do not fit the shared arrays (densities far above the method's).
 */
constexpr int kTileMax = 1024;

__device__ __forceinline__ int spread3(int v)
{
    return (v & 1) | ((v & 2) << 2) | ((v & 4) << 4);
}

__device__ __forceinline__ int morton_key(float4 p, float ox, float oy, float oz, float kx, float ky, float kz)
{
    const int ix = min(7, max(0, (int)((p.x - ox) * kx)));
    const int iy = min(7, max(0, (int)((p.y - oy) * ky)));
    const int iz = min(7, max(0, (int)((p.z - oz) * kz)));
    return spread3(ix) | (spread3(iy) << 1) | (spread3(iz) << 2);
}

/* Sorting key of a coordinate u (from the cell's corner): its float bits, then the caller index, so that keys are
   distinct and their order does not depend on the order in which the cell's entries were placed. */
__device__ __forceinline__ long long tile_key(float u, int x)
{
    return ((long long)__float_as_int(fmaxf(u, 0.f)) << 32) | (unsigned int)x;
}

/* How many of k[lo .. hi) are below ke; lo is a multiple of 8 and k is padded with LLONG_MAX to hi. */
__device__ __forceinline__ int rank_of(const long long* k, int lo, int hi, long long ke)
{
    int r = 0;
    #pragma unroll 2
    for (int f = lo; f < hi; f += 4) {
        const longlong2 v = *reinterpret_cast<const longlong2*>(k + f);
        const longlong2 w = *reinterpret_cast<const longlong2*>(k + f + 2);
        r += v.x < ke;
        r += v.y < ke;
        r += w.x < ke;
        r += w.y < ke;
    }
    return r;
}

/* The CTA's barrier; in the debug build, whether any thread found an index out of range. */
__device__ __forceinline__ bool barrier_bad(bool bad)
{
#ifdef USR_DEBUG_BOUNDS
    return __syncthreads_or(bad) != 0;
#else
    (void)bad;
    __syncthreads();
    return false;
#endif
}

/*
 * The clusters of one cell per CTA, from the cell's entries in any order (k_place): the packing above, the padded
 * layout, each cluster's bounding box; also the descriptor of each of the cell's groups of gcl clusters, and the
 * cell's rows of the pair kernel's fixed-point accumulators (four per slot) set to zero.  The pair kernel, the
 * spreading, the gather and the combination all walk the slots, so an evaluation needs no other order of the atoms.
 * With qsum given, also the charges' sum, from which the spreading takes rho's mean before it splits rho into operand
 * pairs (what the fixed point leaves of the mean is measured and taken off later).
 */
__global__ void __launch_bounds__(256) k_cluster_build(const int* __restrict__ start,
                                                       const int* __restrict__ pstart,
                                                       const int* __restrict__ gfull,
                                                       const int* __restrict__ gpart, int gcl, BoxF b,
                                                       const int* __restrict__ unsorted,
                                                       const float4* __restrict__ wpos,
                                                       int* __restrict__ key, float4* __restrict__ cpos,
                                                       int* __restrict__ cperm, int* __restrict__ ccell,
                                                       float4* __restrict__ bblo, float4* __restrict__ bbhi,
                                                       int4* __restrict__ gdesc,
                                                       unsigned long long* __restrict__ acc,
                                                       ChargeSum* __restrict__ qsum, int n,
                                                       int max_slots, int max_groups, int* __restrict__ status)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    __shared__ __align__(16) long long k0[kTileMax], k1[kTileMax];
    __shared__ long long qwarp[8];
    const int threads = blockDim.x;
    const int c = blockIdx.x;
    const int s0 = start[c], m = start[c + 1] - s0;
    const int p0 = pstart[c], pm = pstart[c + 1] - p0;
    const float unit = qsum ? exp2_int(charge_bits(qsum->max)) : 0.f;
    if (pm == 0) return;                                  // an empty cell has no clusters
    if (!USR_IN_BOUNDS(s0 + m - 1, n, status) || !USR_IN_BOUNDS(p0 + pm - 1, max_slots, status)) return;
    {
        // full groups in cell order, then the partial ones (the pair kernel takes them in that order,
        // so its last work units are the small ones)
        const int f0 = gfull[c], nf = gfull[c + 1] - f0;
        for (int k = threadIdx.x; k < nf; k += threads)
            if (USR_IN_BOUNDS(f0 + k, max_groups, status)) gdesc[f0 + k] = make_int4((p0 >> 3) + k * gcl, c, gcl, 0);
        if (threadIdx.x == 0 && gpart[c + 1] > gpart[c]) {
            const int gp = gfull[b.nc[0] * b.nc[1] * b.nc[2]] + gpart[c];
            if (USR_IN_BOUNDS(gp, max_groups, status))
                gdesc[gp] = make_int4((p0 >> 3) + nf * gcl, c, (pm >> 3) - nf * gcl, 0);
        }
        ulonglong2* a2 = reinterpret_cast<ulonglong2*>(acc + 4 * (size_t)p0);
        for (int e = threadIdx.x; e < 2 * pm; e += threads) a2[e] = make_ulonglong2(0ull, 0ull);
    }
    const int cx = c % b.nc[0], cy = (c / b.nc[0]) % b.nc[1], cz = c / (b.nc[0] * b.nc[1]);
    const float ox = (float)cx / b.cs[0], oy = (float)cy / b.cs[1], oz = (float)cz / b.cs[2];
    // the cell's charges: summed per warp on the first pass, by thread 0 after its barrier (one addition per cell to
    // the one address, and early: an evaluation of 20 k charges takes 1.0 us more than without the sum, 1.5 with it at
    // the kernel's end)
    long long qs = 0;
    auto put_sum = [&]() {
        if (!qsum) return;
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) qs += __shfl_xor_sync(0xffffffffu, qs, o);
        if ((threadIdx.x & 31) == 0) qwarp[threadIdx.x >> 5] = qs;
    };
    auto add_sum = [&]() {
        if (!qsum || threadIdx.x != 0) return;
        for (int w = 1; w < threads >> 5; ++w) qs += qwarp[w];
        atomicAdd(&qsum->sum, (unsigned long long)qs);    // two's complement
    };
    bool bad = false;                                     // (debug build) an entry of the cell is out of range
    if (m <= kTileMax) {
        const int ncl = pm >> 3;
        int sx = 1;                                       // slabs: the cube root of the clusters, rounded
        while ((2 * sx + 1) * (2 * sx + 1) * (2 * sx + 1) <= 8 * ncl) ++sx;
        for (int e = threadIdx.x; e < pm; e += threads) {
            long long key0 = LLONG_MAX;
            if (e < m) {
                const int x = unsorted[s0 + e];
                if (!USR_IN_BOUNDS(x, n, status)) { bad = true; continue; }
                const float4 p = wpos[x];
                key0 = tile_key(p.x - ox, x);
                qs += __float2ll_rn(p.w * unit);
            }
            k0[e] = key0;
        }
        put_sum();
        if (barrier_bad(bad)) return;
        add_sum();
        // each pass puts every atom at its place in the next order and stores its next key there
        for (int e = threadIdx.x; e < pm; e += threads) {
            if (e < m) {
                const long long ke = k0[e];
                const int r = rank_of(k0, 0, pm, ke), x = (int)ke;
                k1[r] = tile_key(wpos[x].y - oy, x);
            } else {
                k1[e] = LLONG_MAX;
            }
        }
        __syncthreads();
        // slab s holds the clusters [ncl s / sx, ncl (s + 1) / sx); column y of its kc clusters likewise
        for (int r = threadIdx.x; r < pm; r += threads) {
            const int s = (((r >> 3) + 1) * sx - 1) / ncl;
            const int a0 = 8 * (ncl * s / sx), a1 = 8 * (ncl * (s + 1) / sx);
            if (r < m) {
                const long long kr = k1[r];
                const int x = (int)kr;
                k0[a0 + rank_of(k1, a0, a1, kr)] = tile_key(wpos[x].z - oz, x);
            } else {
                k0[r] = LLONG_MAX;
            }
        }
        __syncthreads();
        for (int q = threadIdx.x; q < m; q += threads) {
            const int s = (((q >> 3) + 1) * sx - 1) / ncl;
            const int l0 = ncl * s / sx, kc = ncl * (s + 1) / sx - l0;
            int sy = 1;                                   // columns: the square root of the slab's clusters, rounded
            while ((2 * sy + 1) * (2 * sy + 1) <= 4 * kc) ++sy;
            const int y = (((q >> 3) - l0 + 1) * sy - 1) / kc;
            const int b0 = 8 * (l0 + kc * y / sy), b1 = 8 * (l0 + kc * (y + 1) / sy);
            const long long kq = k0[q];
            const int t = b0 + rank_of(k0, b0, b1, kq), x = (int)kq;
            cpos[p0 + t] = wpos[x];
            cperm[p0 + t] = x;
        }
    } else {
        const float fx = 8.0f * b.cs[0], fy = 8.0f * b.cs[1], fz = 8.0f * b.cs[2];
        int* kk = key + s0;
        const int* xs = unsorted + s0;
        for (int e = threadIdx.x; e < m; e += threads) {
            if (!USR_IN_BOUNDS(xs[e], n, status)) { bad = true; continue; }
            const float4 p = wpos[xs[e]];
            kk[e] = morton_key(p, ox, oy, oz, fx, fy, fz);
            qs += __float2ll_rn(p.w * unit);
        }
        put_sum();
        if (barrier_bad(bad)) return;
        add_sum();
        // rank of (Morton code, caller index), four atoms to a thread, against a tile of the cell's keys at a time in
        // shared memory.  Bound: the m^2 comparisons.  Evaluations with 3,000 charges in one cell / 20,000 in eight:
        // 0.33 / 1.87 ms; 2.49 / 12.1 ms with one key at a time from global memory.
        for (int base = 0; base < m; base += 4 * threads) {
            long long ke[4];
            int r[4] = {0, 0, 0, 0};
            #pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = base + u * threads + threadIdx.x;
                ke[u] = e < m ? ((long long)kk[e] << 32) | (unsigned int)xs[e] : LLONG_MIN;
            }
            for (int t0 = 0; t0 < m; t0 += kTileMax) {
                const int tn = min(kTileMax, m - t0), tp = (tn + 1) & ~1;
                __syncthreads();                          // the previous tile has been read
                for (int f = threadIdx.x; f < tp; f += threads)
                    k0[f] = f < tn ? ((long long)kk[t0 + f] << 32) | (unsigned int)xs[t0 + f] : LLONG_MAX;
                __syncthreads();
                #pragma unroll 4
                for (int f = 0; f < tp; f += 2) {
                    const longlong2 v = *reinterpret_cast<const longlong2*>(k0 + f);
                    #pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        r[u] += v.x < ke[u];
                        r[u] += v.y < ke[u];
                    }
                }
            }
            #pragma unroll
            for (int u = 0; u < 4; ++u)
                if (base + u * threads + threadIdx.x < m) {
                    const int x = (int)ke[u];
                    cpos[p0 + r[u]] = wpos[x];
                    cperm[p0 + r[u]] = x;
                }
        }
    }
    for (int e = m + threadIdx.x; e < pm; e += threads) {
        // padding rows: far from the box, so never within r_c of an atom, and 4e4 A apart within
        // a cluster (rows of different cells may coincide; the pair kernel never uses their sums)
        const float far = -1.0e6f - 4.0e4f * (float)(e & 7);
        cpos[p0 + e] = make_float4(far, far, far, 0.0f);
        cperm[p0 + e] = -1;
    }
    __syncthreads();
    // bounding boxes: eight lanes per cluster (pm is a multiple of 8, so a cluster's lanes run together)
    for (int e = threadIdx.x; e < pm; e += threads) {
        float4 lo = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f), hi = make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f);
        if (e < m) {
            const float4 p = cpos[p0 + e];
            lo = make_float4(p.x, p.y, p.z, 0.f);
            hi = lo;
        }
        const unsigned int peers = 0xffu << (threadIdx.x & 24);
        #pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            lo.x = fminf(lo.x, __shfl_xor_sync(peers, lo.x, o));
            lo.y = fminf(lo.y, __shfl_xor_sync(peers, lo.y, o));
            lo.z = fminf(lo.z, __shfl_xor_sync(peers, lo.z, o));
            hi.x = fmaxf(hi.x, __shfl_xor_sync(peers, hi.x, o));
            hi.y = fmaxf(hi.y, __shfl_xor_sync(peers, hi.y, o));
            hi.z = fmaxf(hi.z, __shfl_xor_sync(peers, hi.z, o));
        }
        if ((e & 7) == 0) {
            const int cl = (p0 + e) >> 3;
            bblo[cl] = lo;
            bbhi[cl] = hi;
            ccell[cl] = c;
        }
    }
}

cudaError_t launch_bin(int n, const float4* xyzq, const BoxF& b, int ncell, int* count, int* cell_of, int* slot,
                       float4* wpos, int* cell_start, int* pstart, int* unsorted, int* perm, float4* spos,
                       int* status, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int) * (size_t)ncell, st);
    if (e != cudaSuccess) return e;
    int nb = (n + 255) / 256;
    k_bin_count<<<nb, 256, 0, st>>>(n, xyzq, b, count, cell_of, slot, wpos, nullptr, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_scan<<<1, 1024, 0, st>>>(ncell, count, cell_start, pstart, nullptr, nullptr, 1, nullptr, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_place<<<nb, 256, 0, st>>>(n, cell_of, slot, cell_start, unsorted, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_cell_sort<<<ncell, kSortThreads, 0, st>>>(n, cell_start, unsorted, wpos, perm, spos, status);
    return cudaGetLastError();
}

/* The cell list: counts, scan (with the pair kernel's group counts), placement (any order within a cell). */
void launch_bin_list(int n, const float4* xyzq, const BoxF& b, int ncell, int* count, int* cell_of, int* slot,
                     float4* wpos, int* cell_start, int* pstart, int* gfull, int* gpart, int* queue,
                     ChargeSum* qsum, int* unsorted, int* status, cudaStream_t st)
{
    // count[] is zero on entry: the context zeroes it when it is (re)configured, and k_scan zeroes every
    // entry after reading it, ready for the next evaluation (no memset between the kernels)
    const int gcl = near_group_clusters();
    int nb = (n + 255) / 256;
    launch_pdl(k_bin_count, nb, 256, 0, st, n, xyzq, b, count, cell_of, slot, wpos, qsum, status);
    launch_pdl(k_scan, 1, 1024, 0, st, ncell, count, cell_start, pstart, gfull, gpart, gcl, queue, qsum);
    launch_pdl(k_place, nb, 256, 0, st, n, cell_of, slot, cell_start, unsorted, status);
}

/* Each cell's atoms in the order of their caller indices (the canonical order of the inspection entry points). */
void launch_cell_sort(int n, int ncell, const int* cell_start, const int* unsorted, const float4* wpos, int* perm,
                      float4* spos, int* status, cudaStream_t st)
{
    launch_pdl(k_cell_sort, ncell, kSortThreads, 0, st, n, cell_start, unsorted, wpos, perm, spos, status);
}

/* The clusters from the cell list (slot[] of launch_bin_list is reused for keys). */
void launch_clusters(int n, const BoxF& b, int ncell, const int* cell_start, const int* pstart, const int* gfull,
                     const int* gpart, int4* gdesc, const int* unsorted, const float4* wpos, int* key, float4* cpos,
                     int* cperm, int* ccell, float4* bblo, float4* bbhi, unsigned long long* near_acc,
                     ChargeSum* qsum, int max_clusters, int max_groups, int* status, cudaStream_t st)
{
    // a thread per atom of a mean cell, within 128 and 256
    const int threads = n > 128LL * ncell ? 256 : 128;
    launch_pdl(k_cluster_build, ncell, threads, 0, st, cell_start, pstart, gfull, gpart, near_group_clusters(), b,
               unsorted, wpos, key, cpos, cperm, ccell, bblo, bbhi, gdesc, near_acc, qsum, n, 8 * max_clusters,
               max_groups, status);
}

}  // namespace usr

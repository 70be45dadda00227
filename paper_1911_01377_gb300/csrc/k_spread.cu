/*
 * k_spread.cu -- charge spreading of the far part (the GSE scheme named in Sec. IV.A, Eq. 32's first
 * spreading Gaussian):
 *   rho_g = sum_i q_i exp(-|g - r_i|^2 / (2 sigma_s^2))   (normalisation folded into the convolution scale)
 * written once per grid point, and the grid mean of what was written (rho's k = 0 mode, dropped per Eq. 4; the
 * x pass of the convolutions or the first restriction takes it off).  The split forms take the mean that the net
 * charge gives off rho before they split it.
 *
 * Owner-computes, as a contraction over atoms: a warp owns a brick of 16 x 8 x 8 grid points (x, y, z) and
 * for eight atoms at a time adds the product X YZ_z of their x weights (16 points x 8 atoms, charge included)
 * and their y weights times the z weight of plane z (8 atoms x 8 points) for each of its 8 planes, with the
 * brick's sums in registers.  Two forms:
 *
 *   tensor cores (mma.sync m16n8k8): the split forms (TF32x3 and BF16x3 convolutions) with 8 and 10 points.  The
 *       operands are split into TF32 high and low parts (to nearest) and three products are accumulated in FP32,
 *       which keeps about 22 bits of each factor; the MMA truncates its sums, so a brick's sums carry a bias of
 *       about 1e-7.  The tcgen05 form would need the y-z products in shared memory, 256 bytes per atom and plane;
 *       here they are formed in registers.
 *   FMA: the FP32 form, and every form from 12 points on.  Two-wide FP32 FMAs, a lane four x points of one y in
 *       every plane, in blocks of 16 atoms that are summed apart (a point of a 12-point stencil receives about 170
 *       terms).  The tensor cores' bias does not cancel over the net charge of a region: with them, the far
 *       potential of a drop of water in vacuum (6,000 charges in 90 A) was off by 6.2e-6 of its norm, with FMAs
 *       in one chain by 4.6e-6, with blocks by 1.8e-6, 1.0e-6 of which is the method's own error at 12 points (in
 *       TF32x3 5.0e-6 and 1.8e-6; with 10 points the stencil itself leaves 4e-5).  Evaluations with FMAs / on the
 *       tensor cores: FP32 form, 3,000 charges 72.1 / 72.1 us, 7,013 ions 93.0 / 92.9, slab 273 / 269, 200 k
 *       charges 932 / 908; TF32x3, 60,000 ions at 16 points 344 / 327.  (With more than 128 registers where eight
 *       warps share a brick, small systems take 1 to 2 us less, and 6,400 charges at r_c = 13 A 114 us instead of
 *       103: the pair kernel's CTAs must wait.)
 *
 * Every warp works by itself: it lists the atoms of the cells its brick's stencils can reach (rows of cells,
 * periodic images as separate rows), keeps those that do reach in a small queue in list order, and evaluates
 * the weights of eight of them straight into the operand registers (a lane two x, one y and one z weight of
 * two atoms; the z weights pass through shared memory).  With few bricks, S warps share one: each takes every
 * S-th chunk of the list, and their sums are added in a fixed order at the end.  There are no atomics, no
 * halo and no second pass over tiles, and every point receives its terms in a fixed order.
 *
 * Bound: issue slots and the latency of the list (39 % of the slots used on the slab, whose 320 bricks leave two warps
 * to a scheduler, 59 % for 200 k charges; tensor pipe 21 and 32 % active).  (P + 15) / 16 ((P + 7) / 8)^2 bricks per
 * atom at 44 instructions each, the listing included.  Alone (ncu): 42 us on the slab at r_c = 8 A (P = 8), 115 us
 * for 200 k charges (P = 10), 328 us for 1.06 M (P = 8); FMA form 71 us on the slab (P = 12; 52 % of the slots).
 * The earlier form (shared-memory tiles per block of cells, one read-modify-write per stencil point, then a reduction
 * over overlapping tiles) took 36 + 23 us and 157 + 73 us (141 at P = 12): 940 instructions per atom at P = 10
 * against 310, held by shared-memory wavefronts and by the tiles' 13-fold halo traffic.  Not kept: bricks of a CTA
 * with weight rows shared by its warps, by FP32 FMAs 217 us (the register side of broadcast loads), on the tensor
 * cores 172 us (barriers); FMAs where the stencil does not need them (evaluations of the split forms 1 to 3 % slower,
 * the FP32 pipe is the pair kernel's); the tensor cores with compensated sums of the groups in the FP32 form (the
 * drop's far potential off by 5.7e-6, slab 280 us per evaluation); up to 16 warps per brick on one flattened list
 * (68 -> 65 us per evaluation of 2 k charges, 598 -> 606 us of 200 k).
 */
#include <algorithm>

#include <cuda_bf16.h>

#include "usr_internal.h"

namespace usr {

namespace {

constexpr int kBrickX = 16, kBrick = 8;   // brick extent along x; along y and z
constexpr int kSpreadWarps = 4;           // warps per CTA (8 when eight share a brick)
constexpr int kEnough = 1000;             // warps in all that a launch tries to reach by sharing bricks
constexpr int kQueue = 64;                // queue slots per warp: fewer than 8 waiting, plus one chunk of 32

__device__ __forceinline__ int floor_div(int a, int b)
{
    const int q = a / b;
    return q - (a % b < 0 ? 1 : 0);
}

/* Compensated FP32 sum (Neumaier). */
struct CSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = __fadd_rn(s, x);
        c = __fadd_rn(c, fabsf(s) >= fabsf(x) ? __fadd_rn(__fsub_rn(s, t), x) : __fadd_rn(__fsub_rn(x, t), s));
        s = t;
    }
};

__device__ __forceinline__ double warp_sum(CSum cs)
{
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float s = __shfl_xor_sync(0xffffffffu, cs.s, o), c = __shfl_xor_sync(0xffffffffu, cs.c, o);
        cs.add(s);
        cs.c = __fadd_rn(cs.c, c);
    }
    return (double)cs.s + (double)cs.c;
}

__device__ __forceinline__ double warp_sum(double v)
{
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

/* x to TF32 precision, to nearest (the MMA reads the high 19 bits of its operands). */
__device__ __forceinline__ float tf32_hi(float x)
{
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

/* d += a b: a 16 x 8 (row = lane / 4 (+ 8), k = lane % 4 (+ 4)), b 8 x 8 (k = lane % 4 (+ 4), column = lane / 4),
   d rows lane / 4 (+ 8), columns 2 (lane % 4) (+ 1). */
__device__ __forceinline__ void mma_tf32(float (&d)[4], const float (&a)[4], float b0, float b1)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(__float_as_uint(a[0])), "r"(__float_as_uint(a[1])), "r"(__float_as_uint(a[2])),
                   "r"(__float_as_uint(a[3])), "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)));
}

struct SpreadWarp {
    float4 f[kQueue];        // queue: fractional offsets (x, y, z) and charge
    int b[kQueue];           // the stencil's first point per axis from the brick's, + 32, 8 bits each
    float z[8][kBrick];      // z weights of the current eight atoms
};

/* The FMA form's further weights of the current eight atoms (rows of x weights 24 floats apart: a warp's stores of
   four rows then touch each bank once). */
struct SpreadWeights {
    float x[8][kBrickX + 8];
    float y[8][kBrick];
};

template <int S, int WARPS, bool FMA>
struct SpreadShared {
    SpreadWarp w[WARPS];
    SpreadWeights xy[FMA ? WARPS : 1];
    float4 share[S > 1 ? (WARPS - WARPS / S) * 256 : 1];   // bricks' shares of the splits after the first
    double red[WARPS];
    int is_last;
};

}  // namespace

/* out: 0 FP32 rho; 1 and 2 the operand split of the tensor-core convolutions, rho = hi + lo with hi rounded to
   TF32 (1) or BF16 (2).  rho32: FP32 copy beside a split (may be null). */
template <int S, int WARPS, bool FMA>
__global__ void __launch_bounds__(32 * WARPS, 16 / WARPS) k_spread(const float4* __restrict__ pos,
                                                        const int* __restrict__ pstart, GridArgs g, int P,
                                                        int bricks_x, int bricks_y, int bricks, int out,
                                                        const ChargeSum* __restrict__ qsum,
                                                        void* __restrict__ rho, void* __restrict__ rho_lo,
                                                        float* __restrict__ rho32, double* __restrict__ partial,
                                                        unsigned int* __restrict__ counter,
                                                        double* __restrict__ mean, int* __restrict__ status)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    constexpr int NB = WARPS / S;
    __shared__ __align__(16) SpreadShared<S, WARPS, FMA> sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int H = P / 2;
    const int n0 = g.box.n[0], n1 = g.box.n[1], n2 = g.box.n[2];
    const int ncx = g.box.nc[0], ncy = g.box.nc[1], ncz = g.box.nc[2];
    // this warp's brick and its share of the list
    const int split = warp / NB, brick = blockIdx.x * NB + warp % NB;
    const bool owns = brick < bricks;
    const int ox = brick % bricks_x * kBrickX, oy = brick / bricks_x % bricks_y * kBrick,
              oz = brick / (bricks_x * bricks_y) * kBrick;
    const int ex = min(kBrickX, n0 - ox), ey = min(kBrick, n1 - oy), ez = min(kBrick, n2 - oz);
    const int tq = lane & 3, gq = lane >> 2;             // thread and group of the MMA fragments
    SpreadWarp& W = sh.w[warp];
    // exp(-d^2 hh) = 2^(d^2 c)
    const float kl = -1.4426950408889634f;
    const float cx = g.hh[0] * kl, cy = g.hh[1] * kl, cz = g.hh[2] * kl;
    // per plane z, the points (x, y): (gq, 2 tq), (gq, 2 tq + 1), (gq + 8, 2 tq), (gq + 8, 2 tq + 1); FMA: (4 tq, gq)
    // .. (4 tq + 3, gq), acc holds the atoms since the last fold into sum
    float acc[8][4], sum[FMA ? 8 : 1][4];
    int groups = 0;
    #pragma unroll
    for (int z = 0; z < 8; ++z)
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[z][k] = 0.f;
            if (FMA) sum[z][k] = 0.f;
        }

    // add `nb` <= 8 atoms from the queue's head to the brick
    auto add8 = [&](int head, int nb) {
        // atoms tq and tq + 4 (past the end: the first one again, with charge 0)
        const int ia = (head + (tq < nb ? tq : 0)) & (kQueue - 1), ib = (head + (tq + 4 < nb ? tq + 4 : 0)) & (kQueue - 1);
        const float4 fa = W.f[ia], fb = W.f[ib];
        const int pa = W.b[ia], pb = W.b[ib];
        const float qa = tq < nb ? fa.w : 0.f, qb = tq + 4 < nb ? fb.w : 0.f;
        // weight of the point at offset i from the brick for a stencil that starts at b (8 bits of p, + 32)
        auto weight = [&](int i, int p, int sh8, float t, float c) {
            const int k = i + 32 - ((p >> sh8) & 255);
            const float d = (float)(k - H + 1) - t;
            float w;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(d * d * c));
            return (unsigned int)k < (unsigned int)P ? w : 0.f;
        };
        W.z[tq][gq] = weight(gq, pa, 16, fa.z, cz);
        W.z[tq + 4][gq] = weight(gq, pb, 16, fb.z, cz);
        const float x[4] = {qa * weight(gq, pa, 0, fa.x, cx), qa * weight(gq + 8, pa, 0, fa.x, cx),
                            qb * weight(gq, pb, 0, fb.x, cx), qb * weight(gq + 8, pb, 0, fb.x, cx)};
        const float ya = weight(gq, pa, 8, fa.y, cy), yb = weight(gq, pb, 8, fb.y, cy);
        if (FMA) {
            SpreadWeights& U = sh.xy[warp];
            U.x[tq][gq] = x[0];
            U.x[tq][gq + 8] = x[1];
            U.x[tq + 4][gq] = x[2];
            U.x[tq + 4][gq + 8] = x[3];
            U.y[tq][gq] = ya;
            U.y[tq + 4][gq] = yb;
            __syncwarp();
            #pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float4 wx = *reinterpret_cast<const float4*>(&U.x[k][4 * tq]);
                const float wy = U.y[k][gq];
                const float2 w0 = __fmul2_rn(make_float2(wx.x, wx.y), make_float2(wy, wy));
                const float2 w1 = __fmul2_rn(make_float2(wx.z, wx.w), make_float2(wy, wy));
                const float4 za = *reinterpret_cast<const float4*>(&W.z[k][0]);
                const float4 zb = *reinterpret_cast<const float4*>(&W.z[k][4]);
                const float wz[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
                #pragma unroll
                for (int z = 0; z < 8; ++z) {
                    const float2 zz = make_float2(wz[z], wz[z]);
                    const float2 r0 = __ffma2_rn(w0, zz, make_float2(acc[z][0], acc[z][1]));
                    const float2 r1 = __ffma2_rn(w1, zz, make_float2(acc[z][2], acc[z][3]));
                    acc[z][0] = r0.x;
                    acc[z][1] = r0.y;
                    acc[z][2] = r1.x;
                    acc[z][3] = r1.y;
                }
            }
            __syncwarp();
            if ((++groups & 1) == 0)
                #pragma unroll
                for (int z = 0; z < 8; ++z)
                    #pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const float2 r = __fadd2_rn(make_float2(sum[z][k], sum[z][k + 1]),
                                                    make_float2(acc[z][k], acc[z][k + 1]));
                        sum[z][k] = r.x;
                        sum[z][k + 1] = r.y;
                        acc[z][k] = acc[z][k + 1] = 0.f;
                    }
            return;
        }
        float xh[4], xl[4];
        #pragma unroll
        for (int k = 0; k < 4; ++k) {
            xh[k] = tf32_hi(x[k]);
            xl[k] = x[k] - xh[k];
        }
        __syncwarp();
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 za = *reinterpret_cast<const float4*>(&W.z[tq][4 * h]);
            const float4 zb = *reinterpret_cast<const float4*>(&W.z[tq + 4][4 * h]);
            const float z0[4] = {za.x, za.y, za.z, za.w}, z1[4] = {zb.x, zb.y, zb.z, zb.w};
            #pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float p0 = ya * z0[k], p1 = yb * z1[k];
                const float h0 = tf32_hi(p0), h1 = tf32_hi(p1);
                // the MMA truncates its sums: each group's is formed apart, small products first, and added to
                // the brick's to nearest (chaining the groups in the MMA shrank rho by 2e-6)
                float t[4] = {0.f, 0.f, 0.f, 0.f};
                mma_tf32(t, xl, h0, h1);
                mma_tf32(t, xh, p0 - h0, p1 - h1);
                mma_tf32(t, xh, h0, h1);
                #pragma unroll
                for (int c = 0; c < 4; ++c) acc[4 * h + k][c] += t[c];
            }
        }
        __syncwarp();
    };

    if (owns) {
        int c0[3], c1[3];                                 // cells that may hold atoms whose stencil reaches the brick
        {
            const int o[3] = {ox, oy, oz}, e[3] = {ex, ey, ez};
            #pragma unroll
            for (int a = 0; a < 3; ++a)
                spread_cells(o[a], e[a], H, g.box.n[a], g.box.nc[a], kSpreadMargin, &c0[a], &c1[a]);
        }
        const int ny = c1[1] - c0[1] + 1, nz = c1[2] - c0[2] + 1;
        const int px = floor_div(c0[0], ncx), npx = floor_div(c1[0], ncx) - px + 1;   // periods the x range touches
        const int runs = nz * ny * npx;
        int head = 0, count = 0, turn = 0;
        for (int rb = 0; rb < runs; rb += 32) {
            // lane = one run of cells: its first slot, length and image shift (grid points, from the brick)
            int first = 0, cnt = 0, sx = 0, sy = 0, sz = 0;
            const int id = rb + lane;
            if (id < runs) {
                const int cyu = c0[1] + id / npx % ny, czu = c0[2] + id / (npx * ny), kx = px + id % npx;
                const int qy = floor_div(cyu, ncy), qz = floor_div(czu, ncz);
                const int row = ((czu - qz * ncz) * ncy + (cyu - qy * ncy)) * ncx;
                first = pstart[row + max(c0[0] - kx * ncx, 0)];
                cnt = pstart[row + min(c1[0] - kx * ncx, ncx - 1) + 1] - first;
                sx = kx * n0 - ox - H + 1;
                sy = qy * n1 - oy - H + 1;
                sz = qz * n2 - oz - H + 1;
            }
            const int here = min(32, runs - rb);
            for (int r = 0; r < here; ++r) {
                const int rc = __shfl_sync(0xffffffffu, cnt, r), rf = __shfl_sync(0xffffffffu, first, r);
                if (rc == 0) continue;
                const int rx = __shfl_sync(0xffffffffu, sx, r), ry = __shfl_sync(0xffffffffu, sy, r);
                const int rz = __shfl_sync(0xffffffffu, sz, r);
                // this warp's chunks of 32 atoms: every S-th of the list
                int base = 32 * ((split - turn) & (S - 1));
                turn += (rc + 31) >> 5;
                // atom k of the run; past its end a padding slot (these lie near -1e6)
                auto fetch = [&](int k) {
                    return k < rc && USR_IN_BOUNDS(rf + k, g.max_slots, status) ? pos[rf + k]
                                                                                : make_float4(-1.0e6f, 0.f, 0.f, 0.f);
                };
                float4 next = fetch(base + lane);
                for (; base < rc; base += 32 * S) {
                    const float4 p = next;
                    bool ok = p.x > -5.0e5f;
                    next = fetch(base + 32 * S + lane);
                    const float ux = p.x * g.box.gs[0], uy = p.y * g.box.gs[1], uz = p.z * g.box.gs[2];
                    const float fx = floorf(ux), fy = floorf(uy), fz = floorf(uz);
                    const int b0 = (int)fx + rx, b1 = (int)fy + ry, b2 = (int)fz + rz;
                    ok = ok && b0 > -P && b0 < ex && b1 > -P && b1 < ey && b2 > -P && b2 < ez;
                    const unsigned int bal = __ballot_sync(0xffffffffu, ok);
                    if (ok) {
                        const int q = (head + count + __popc(bal & ((1u << lane) - 1u))) & (kQueue - 1);
                        // (BF16 operands keep nothing of the fraction's last digits)
                        W.f[q] = out == 2 ? make_float4(ux - fx, uy - fy, uz - fz, p.w)
                                          : make_float4(grid_frac(g.box, 0, p.x, fx), grid_frac(g.box, 1, p.y, fy),
                                                        grid_frac(g.box, 2, p.z, fz), p.w);
                        W.b[q] = (b0 + 32) | (b1 + 32) << 8 | (b2 + 32) << 16;
                    }
                    count += __popc(bal);
                    __syncwarp();
                    while (count >= 8) {
                        add8(head, 8);
                        head = (head + 8) & (kQueue - 1);
                        count -= 8;
                    }
                }
            }
        }
        if (count > 0) add8(head, count);
    }
    // The operand splits keep a fixed number of digits of what they are given: rho's mean (the net charge over the
    // grid, dropped as the k = 0 mode) is taken off before.  Any constant would do; the mean of what is written is
    // measured below, and the x pass (or the first restriction) takes it off exactly.
    const float m0 = out == 0 ? 0.f : __ll2float_rn((long long)qsum->sum) * exp2_int(-charge_bits(qsum->max)) * g.qmean;
    if (FMA)
        #pragma unroll
        for (int z = 0; z < 8; ++z)
            #pragma unroll
            for (int k = 0; k < 4; ++k) acc[z][k] += sum[z][k];

    if (S > 1) {
        // add the bricks' shares in order of the split
        if (split > 0)
            #pragma unroll
            for (int z = 0; z < 8; ++z)
                sh.share[((warp - NB) * 8 + z) * 32 + lane] = make_float4(acc[z][0], acc[z][1], acc[z][2], acc[z][3]);
        __syncthreads();
        if (split == 0)
            for (int s = 1; s < S; ++s)
                #pragma unroll
                for (int z = 0; z < 8; ++z) {
                    const float4 v = sh.share[(((s - 1) * NB + warp) * 8 + z) * 32 + lane];
                    acc[z][0] += v.x;
                    acc[z][1] += v.y;
                    acc[z][2] += v.z;
                    acc[z][3] += v.w;
                }
    }
    CSum cs;
    if (split == 0 && owns) {
        #pragma unroll
        for (int z = 0; z < 8; ++z)
            #pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int x = FMA ? 4 * tq + k : gq + 8 * (k >> 1), y = FMA ? gq : 2 * tq + (k & 1);
                if (x >= ex || y >= ey || z >= ez) continue;
                const size_t i = ((size_t)(oz + z) * n1 + (oy + y)) * n0 + (ox + x);
                const float v = acc[z][k] - m0;
                cs.add(v);
                if (out == 0) {
                    static_cast<float*>(rho)[i] = v;
                } else if (out == 1) {
                    uint32_t hb;
                    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hb) : "f"(v));
                    const float hi = __uint_as_float(hb);
                    static_cast<float*>(rho)[i] = hi;
                    static_cast<float*>(rho_lo)[i] = v - hi;
                } else {
                    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
                    static_cast<__nv_bfloat16*>(rho)[i] = hi;
                    static_cast<__nv_bfloat16*>(rho_lo)[i] = __float2bfloat16_rn(v - __bfloat162float(hi));
                }
                if (out != 0 && rho32) rho32[i] = v;
            }
    }
    const double local = warp_sum(cs);
    if (lane == 0) sh.red[warp] = local;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int w = 0; w < WARPS; ++w) s += sh.red[w];
        partial[blockIdx.x] = s;
        __threadfence();
        sh.is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (sh.is_last) {
        // grid mean from the CTAs' sums, in order (the same whichever CTA is last)
        __threadfence();
        double s = 0.0;
        for (int k = tid; k < (int)gridDim.x; k += 32 * WARPS) s += ((volatile double*)partial)[k];
        s = warp_sum(s);
        __syncthreads();
        if (lane == 0) sh.red[warp] = s;
        __syncthreads();
        if (tid == 0) {
            double tot = 0.0;
            for (int w = 0; w < WARPS; ++w) tot += sh.red[w];
            *mean = tot / ((double)n0 * n1 * n2);
            *counter = 0u;
        }
    }
}

/* out = rho - mean (the virial's grid products want rho without its k = 0 mode). */
__global__ void __launch_bounds__(256) k_sub_mean(long long G, const float* rho, float* out, const double* __restrict__ mean)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    const float m = (float)*mean;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < G; i += (long long)gridDim.x * 256)
        out[i] = rho[i] - m;
}

void launch_sub_mean(long long G, const float* rho, float* out, const double* mean, cudaStream_t st)
{
    launch_pdl(k_sub_mean, (unsigned)std::min<long long>((G + 255) / 256, 4 * 152), 256, 0, st, G, rho, out, mean);
}

/* ------------------------------------------------------------------ launch */

namespace {

inline int bricks_along(int n, int e) { return (n + e - 1) / e; }

int bricks_of(const int* n) { return bricks_along(n[0], kBrickX) * bricks_along(n[1], kBrick) * bricks_along(n[2], kBrick); }

/*
 * Warps per brick: the fewest that give kEnough warps in all, at most 8.  Sharing shortens the list each warp
 * works through and adds a pass over the shares; measured per evaluation with 1000 / 2000 / 4000 warps: slab
 * (320 bricks) 165 / 169 / 169 us at r_c = 8 A and 321 / 327 / 326 us in the tight form; 200 k charges (2,048
 * bricks) 627 / 624 / 652 us.
 */
int splits_of(const int* n)
{
    int s = 1;
    while (s < 8 && (long long)bricks_of(n) * s < kEnough) s *= 2;
    return s;
}

/* CTAs of 4 warps: 16 k registers, the slot that the pair kernel leaves free on an SM (1.06 M charges: 2.52 ms per
   evaluation against 2.63 with 8). */
int warps_of(int s) { return s == 8 ? 8 : kSpreadWarps; }

}  // namespace

int spread_ctas(const int* n)
{
    const int s = splits_of(n), nb = warps_of(s) / s;
    return (bricks_of(n) + nb - 1) / nb;
}

void launch_spread(int P, const ClusterList& L, const GridArgs& g, int split, const ChargeSum* qsum, void* rho,
                   void* rho_lo, float* rho32, double* partial, unsigned int* counter, double* mean, int* status,
                   cudaStream_t st)
{
    const int bx = bricks_along(g.box.n[0], kBrickX), by = bricks_along(g.box.n[1], kBrick);
    const bool fma = split == 0 || P >= 12;   // 12 points and more resolve what the tensor cores' sums lack (above)
#define USR_SPREAD_FORM(S, W, F)                                                                                   \
    launch_pdl(k_spread<S, W, F>, spread_ctas(g.box.n), 32 * W, 0, st, L.cpos, L.pstart, g, P, bx, by,              \
               bricks_of(g.box.n), split, qsum, rho, rho_lo, rho32, partial, counter, mean, status)
#define USR_SPREAD(S, W) if (fma) USR_SPREAD_FORM(S, W, true); else USR_SPREAD_FORM(S, W, false)
    switch (splits_of(g.box.n)) {
        case 1: USR_SPREAD(1, kSpreadWarps); break;
        case 2: USR_SPREAD(2, kSpreadWarps); break;
        case 4: USR_SPREAD(4, kSpreadWarps); break;
        default: USR_SPREAD(8, 8); break;
    }
#undef USR_SPREAD
#undef USR_SPREAD_FORM
}

}  // namespace usr

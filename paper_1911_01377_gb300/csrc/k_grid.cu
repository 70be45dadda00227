/*
 * k_grid.cu -- the gather leg of the far part (Sec. V with Gaussian spreading,
 * the GSE scheme named in Sec. IV.A; the spreading leg is k_spread.cu) and the
 * combination with the near part, atomic-free and deterministic.
 *
 *   gather   phi_far,i = sum_g w(g - r_i) psi_g and F_far,i = -q_i grad phi_far,i
 *            (the second spreading Gaussian of Eq. 32's 1/|S(k)|^2), per cluster
 *            slot, reading psi from global memory; contracts the stencil
 *            separably (z first, per (x, y) column); also psi's grid mean.
 *   combine  after the pair kernel: near + far + the self term -F(0) q_i in
 *            caller order, and E = 1/2 sum q_i phi_i and its parts
 *            (compensated FP32 within a warp, FP64 across warps and blocks).
 */
#include <algorithm>
#include <climits>

#include "usr_internal.h"

namespace usr {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ double warp_sum_d(double v)
{
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

/*
 * Compensated FP32 accumulation (Neumaier): s + c carries the sum to about FP32 rounding of the total,
 * independent of the number of terms.  FP64 is kept for the sums across threads: GB300's FP64 rate is
 * about 1/64 of FP32, so per-element FP64 arithmetic in these kernels cost more than their FP32 work.
 */
struct CSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float t = __fadd_rn(s, x);
        c = __fadd_rn(c, fabsf(s) >= fabsf(x) ? __fadd_rn(__fsub_rn(s, t), x) : __fadd_rn(__fsub_rn(x, t), s));
        s = t;
    }
    // a * b exactly, as the rounded product and its rounding error (fmaf gives the error exactly)
    __device__ __forceinline__ void add_product(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        add(p);
        add(fmaf(a, b, -p));
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

/* A compensated sum over the warp (xor butterfly, FP32 with the error terms carried), as FP64: one conversion
   per warp instead of five FP64 additions per thread (GB300's FP64 pipe is narrow). Callers use lane 0's value. */
__device__ __forceinline__ double warp_sum_c(CSum cs)
{
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float s = __shfl_xor_sync(0xffffffffu, cs.s, o), c = __shfl_xor_sync(0xffffffffu, cs.c, o);
        cs.add(s);
        cs.c = __fadd_rn(cs.c, c);
    }
    return cs.value();
}

/* Periodic wrap of a grid index that lies within two periods of [0, n). */
__device__ __forceinline__ int wrap_once(int v, int n)
{
    if (v < 0) v += n;
    while (v >= n) v -= n;
    return v;
}

}  // namespace

/*
 * out = scale * sum_g a_g b_g (the virial's products of rho with the strain derivatives of psi): compensated FP32
 * within a thread, FP64 partial sums per CTA in a fixed order, the last CTA finishes.
 */
__global__ void __launch_bounds__(256) k_grid_dot(long long G, const float* __restrict__ a,
                                                  const float* __restrict__ b, double scale,
                                                  double* __restrict__ partial, unsigned int* __restrict__ counter,
                                                  double* __restrict__ out)
{
    __shared__ double red[8];
    __shared__ int is_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CSum cs;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < G; i += (long long)gridDim.x * 256)
        cs.add_product(a[i], b[i]);
    double s = warp_sum_c(cs);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        partial[blockIdx.x] = t;
        __threadfence();
        is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (is_last) {
        __threadfence();
        double t = 0.0;
        for (int k = threadIdx.x; k < (int)gridDim.x; k += 256) t += ((volatile double*)partial)[k];
        t = warp_sum_d(t);
        if (lane == 0) red[warp] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            double u = 0.0;
            for (int w = 0; w < 8; ++w) u += red[w];
            *out = u * scale;
            *counter = 0u;
        }
    }
}

void launch_grid_dot(const GridArgs& g, const float* a, const float* b, double scale, double* partial,
                     unsigned int* counter, double* out, cudaStream_t st)
{
    const long long G = (long long)g.box.n[0] * g.box.n[1] * g.box.n[2];
    k_grid_dot<<<kGridDotBlocks, 256, 0, st>>>(G, a, b, scale, partial, counter, out);
}

/*
 * W = W_near + delta E_far + 1/2 <rho, psi_ab>: near from the pair kernel's per-unit slots (the unit count
 * follows from the group totals of the cell list; every thread sums its units in order, then the threads in a
 * fixed tree), far from the six grid dot products (already halved) and E_far.
 */
__global__ void __launch_bounds__(1024) k_virial_finalize(const double* __restrict__ near_w, ClusterList L, int ncell,
                                                          int nsplit, const double* __restrict__ dots,
                                                          const double* __restrict__ energy, double* __restrict__ W)
{
    __shared__ double red[32][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int units = nsplit * (L.gfull[ncell] + L.gpart[ncell]);
    double wn[6] = {0, 0, 0, 0, 0, 0};
    for (int w = threadIdx.x; w < units; w += 1024)
        for (int c = 0; c < 6; ++c) wn[c] += near_w[6 * (size_t)w + c];
    for (int c = 0; c < 6; ++c) {
        const double v = warp_sum_d(wn[c]);
        if (lane == 0) red[warp][c] = v;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double ef = energy[2];
    double t[6];
    for (int c = 0; c < 6; ++c) {
        double v = 0.0;
        for (int w = 0; w < 32; ++w) v += red[w][c];
        t[c] = v + dots[c] + (c < 3 ? ef : 0.0);
    }
    const int map[9] = {0, 3, 4, 3, 1, 5, 4, 5, 2};
    for (int e = 0; e < 9; ++e) W[e] = t[map[e]];
}

void launch_virial_finalize(const double* near_w, const ClusterList& L, int ncell, const double* dots,
                            const double* energy, double* W, cudaStream_t st)
{
    k_virial_finalize<<<1, 1024, 0, st>>>(near_w, L, ncell, near_splits(), dots, energy, W);
}

/* ------------------------------------------------------------------ gather */

/* The pair kernel's near part of a cluster slot: four fixed-point sums (2^-32 units; component c of slot t of a
   cluster at 8 c + t) as FP32. */
__device__ __forceinline__ float4 near_part(const unsigned long long* __restrict__ acc, int slot)
{
    const unsigned long long* a = acc + 32 * (size_t)(slot >> 3) + (slot & 7);
    constexpr float k = 2.3283064365386963e-10f;   // 2^-32, exact
    return make_float4(__ll2float_rn((long long)a[0]) * k, __ll2float_rn((long long)a[8]) * k,
                       __ll2float_rn((long long)a[16]) * k, __ll2float_rn((long long)a[24]) * k);
}

/*
 * Far part at every cluster slot (the gather of Sec. V: the spreading Gaussian of the atom against psi,
 * and its gradient), read straight from psi in global memory: consecutive slots are neighbours in
 * space, so a CTA's stencils overlap and hit in L1 / L2.  A CTA takes consecutive slots, gather_lanes(P)
 * lanes per atom: lane u takes the stencil columns x = u, u + lanes, ... of every row, contracting z first,
 * so the lanes of an atom read one contiguous run of a row per load.  Writes far4[s] = (-q grad phi, phi
 * before the k = 0 correction); the CTAs also sum psi, and the last one writes its mean.
 */
#ifndef USR_GATHER_MINB
#define USR_GATHER_MINB 2   // CTAs per SM the 8- and 10-point gathers are compiled for (3 spills; measured slower)
#endif
constexpr int kGThreads = USR_GATHER_THREADS;   // gather CTA size
constexpr int kGWarps = kGThreads / 32;
#ifndef USR_GATHER_LANES
#define USR_GATHER_LANES 0   // lanes per atom; 0: 5 for P = 10 (two columns each), else 4
#endif
__host__ __device__ constexpr int gather_lanes(int P)
{
    return USR_GATHER_LANES ? USR_GATHER_LANES : (P == 10 ? 5 : 4);
}

/* The CTAs' shares of psi's grid sum in a fixed order (the last CTA), then its mean. */
__device__ __forceinline__ void finish_psi_mean(CSum ps, long long G, double* __restrict__ partial,
                                                unsigned int* __restrict__ counter, double* __restrict__ psi_mean)
{
    __shared__ double red[kGWarps];
    __shared__ int is_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double t = warp_sum_c(ps);
    if (lane == 0) red[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < kGWarps; ++w) v += red[w];
        partial[blockIdx.x] = v;
        __threadfence();
        is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double a = 0.0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += kGThreads) a += ((volatile double*)partial)[k];
    a = warp_sum_d(a);
    __syncthreads();
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < kGWarps; ++w) v += red[w];
        *psi_mean = v / (double)G;
        *counter = 0u;
    }
}

template <int P>
__global__ void __launch_bounds__(kGThreads, (P <= 10 ? USR_GATHER_MINB : 2) * 256 / kGThreads)
    k_gather(const float4* __restrict__ cpos, const int* __restrict__ nslots, const float* __restrict__ psi, GridArgs g,
             float4* __restrict__ far4, double* __restrict__ partial, unsigned int* __restrict__ counter,
             double* __restrict__ psi_mean, int* __restrict__ status)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    constexpr int H = P / 2;
    constexpr int LPA = gather_lanes(P);       // lanes per atom
    constexpr int NC = (P + LPA - 1) / LPA;    // stencil columns per lane
    constexpr int APW = 32 / LPA;              // atoms per warp pass
    constexpr int APC = kGWarps * APW;         // atoms per CTA pass
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slot = lane / LPA, u = lane % LPA;
    const int n0 = g.box.n[0], n1 = g.box.n[1], n2 = g.box.n[2];
    const long long plane = (long long)n0 * n1;
    // psi's mean (its rounding-level k = 0 mode): this CTA's share of the grid sum first
    CSum ps;
    const long long G = plane * n2;
    for (long long i = (long long)blockIdx.x * kGThreads + threadIdx.x; i < G; i += (long long)gridDim.x * kGThreads)
        ps.add(psi[i]);
    const int ns = *nslots;
    for (int s0 = blockIdx.x * APC + warp * APW; s0 < ns; s0 += gridDim.x * APC) {
        const int s = s0 + slot;
        // lanes past APW x LPA hold no atom, and neither do the padding slots (near -1e6)
        float4 p = slot < APW && s < ns && USR_IN_BOUNDS(s, g.max_slots, status) ? cpos[s]
                                                                                 : make_float4(-1.0e6f, 0.f, 0.f, 0.f);
        const bool have = p.x > -5.0e5f;
        if (!have) p = make_float4(0.f, 0.f, 0.f, 0.f);
        const float pc[3] = {p.x, p.y, p.z};
        int base[3];
        float tt[3];
        #pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float uu = pc[a] * g.box.gs[a];
            const float f = floorf(uu);
            tt[a] = grid_frac(g.box, a, pc[a], f);
            base[a] = (int)f - H + 1;
        }
        float wz[P], dz[P], wx[NC], dx[NC];
        int zi[P], xo[NC];
        #pragma unroll
        for (int k = 0; k < P; ++k) {
            const float d2 = (float)(k - H + 1) - tt[2];
            wz[k] = __expf(-d2 * d2 * g.hh[2]);
            dz[k] = wz[k] * d2 * g.dfac[2];
            zi[k] = wrap_once(base[2] + k, n2);
        }
        #pragma unroll
        for (int m = 0; m < NC; ++m) {
            const int c = u + LPA * m;
            const float d0 = (float)(c - H + 1) - tt[0];
            wx[m] = c < P ? __expf(-d0 * d0 * g.hh[0]) : 0.f;
            dx[m] = wx[m] * d0 * g.dfac[0];
            xo[m] = wrap_once(base[0] + (c < P ? c : 0), n0);
        }
        float aphi = 0.f, ax = 0.f, ay = 0.f, az = 0.f;
        #pragma unroll
        for (int jy = 0; jy < P; ++jy) {
            const float d1 = (float)(jy - H + 1) - tt[1];
            const float wy = __expf(-d1 * d1 * g.hh[1]);
            const float dy = wy * d1 * g.dfac[1];
            const int yo = wrap_once(base[1] + jy, n1) * n0;
            float r0 = 0.f, r1 = 0.f, r2 = 0.f;
            #pragma unroll
            for (int m = 0; m < NC; ++m) {
                if (u + LPA * m >= P) continue;
                const float* col = psi + yo + xo[m];
                float v[P];
                #pragma unroll
                for (int k = 0; k < P; ++k) v[k] = __ldg(col + (long long)zi[k] * plane);
                float c0a = 0.f, c0b = 0.f, c1a = 0.f, c1b = 0.f;
                #pragma unroll
                for (int k = 0; k < P; k += 2) {
                    c0a = fmaf(wz[k], v[k], c0a);
                    c1a = fmaf(dz[k], v[k], c1a);
                    c0b = fmaf(wz[k + 1], v[k + 1], c0b);
                    c1b = fmaf(dz[k + 1], v[k + 1], c1b);
                }
                const float cz0 = c0a + c0b, cz1 = c1a + c1b;
                r0 = fmaf(wx[m], cz0, r0);
                r1 = fmaf(dx[m], cz0, r1);
                r2 = fmaf(wx[m], cz1, r2);
            }
            aphi = fmaf(wy, r0, aphi);
            ax = fmaf(wy, r1, ax);
            ay = fmaf(dy, r0, ay);
            az = fmaf(wy, r2, az);
        }
        // the lanes of an atom hold disjoint partial sums: a butterfly for a power of two, else lane u = 0
        // adds those of u = 1, 2, ... in order
        if ((LPA & (LPA - 1)) == 0) {
            #pragma unroll
            for (int o = 1; o < LPA; o <<= 1) {
                aphi += __shfl_xor_sync(0xffffffffu, aphi, o);
                ax += __shfl_xor_sync(0xffffffffu, ax, o);
                ay += __shfl_xor_sync(0xffffffffu, ay, o);
                az += __shfl_xor_sync(0xffffffffu, az, o);
            }
        } else {
            const float p0 = aphi, p1 = ax, p2 = ay, p3 = az;
            #pragma unroll
            for (int o = 1; o < LPA; ++o) {
                aphi += __shfl_down_sync(0xffffffffu, p0, o);
                ax += __shfl_down_sync(0xffffffffu, p1, o);
                ay += __shfl_down_sync(0xffffffffu, p2, o);
                az += __shfl_down_sync(0xffffffffu, p3, o);
            }
        }
        if (have && u == 0) {
            const float qi = p.w;
            far4[s] = make_float4(-qi * ax, -qi * ay, -qi * az, aphi);
        }
    }
    finish_psi_mean(ps, G, partial, counter, psi_mean);
}

/*
 * The gather of the wide stencils (12 points and more) on an even x extent: one warp per atom.  A lane holds two
 * neighbouring x points, aligned (the stencil's points plus zero weights at its ends: NP lanes cover a row), of the
 * rows y = r, r + R, ... (R = 32 / NP rows side by side); it contracts z first, all of a lane's loads
 * independent, then its x points and rows; the warp sums the lanes at the end.  The z weights come from
 * shared memory (lane k evaluates weight k), the x and y weights are the lane's own.
 *
 * Bound: L1 wavefronts (68 % of their peak on the slab; k_gather 56 % at 8 points there and 81 % at 10 for 200 k
 * charges): the rows of a load fall on overlapping banks.  A row is one two-wide load where k_gather spreads each
 * load over 8 atoms' rows: alone on the slab (12 points) 90 -> 76 us.  With 10 points the two are
 * equal (130 against 124 us for 200 k charges) and with 8, four points to a lane, this form is slower (44 against
 * 35 us on the slab): the weights then cost more than the rows.
 */
template <int P>
struct GatherShape {
    static constexpr int NP = (P + 2) / 2;                        // lanes per row: P points at any offset mod 2
    static constexpr int R = 32 / NP < P ? 32 / NP : P;           // rows side by side
    static constexpr int BL = (P + R - 1) / R;                    // rows per lane
};

template <int P>
__global__ void __launch_bounds__(kGThreads, 8)
    k_gather_wide(const float4* __restrict__ cpos, const int* __restrict__ nslots, int per,
                  const float* __restrict__ psi, GridArgs g, float4* __restrict__ far4, double* __restrict__ partial,
                  unsigned int* __restrict__ counter, double* __restrict__ psi_mean, int* __restrict__ status)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    constexpr int H = P / 2;
    typedef GatherShape<P> Sh;
    __shared__ float2 zw[kGWarps][P];          // z weight and its derivative factor
    __shared__ unsigned int zo[kGWarps][P];    // offset of the plane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n0 = g.box.n[0], n1 = g.box.n[1], n2 = g.box.n[2];
    const unsigned int plane = (unsigned int)n0 * n1;
    // psi's mean (its rounding-level k = 0 mode): this CTA's share of the grid sum first
    CSum ps;
    const long long G = (long long)plane * n2;
    for (long long i = (long long)blockIdx.x * kGThreads + threadIdx.x; i < G; i += (long long)gridDim.x * kGThreads)
        ps.add(psi[i]);
    const int slot = lane % Sh::NP, row = lane / Sh::NP;
    const int ns = *nslots;
    for (int c0 = blockIdx.x * (kGWarps * per); c0 < ns; c0 += gridDim.x * (kGWarps * per)) {
        const int s1 = min(ns, c0 + kGWarps * per);
        for (int s = c0 + warp; s < s1; s += kGWarps) {
            if (!USR_IN_BOUNDS(s, g.max_slots, status)) continue;
            const float4 p = cpos[s];
            if (p.x < -5.0e5f) continue;           // a padding slot (near -1e6)
            const float ux = p.x * g.box.gs[0], uy = p.y * g.box.gs[1], uz = p.z * g.box.gs[2];
            const float fx = floorf(ux), fy = floorf(uy), fz = floorf(uz);
            const int b0 = (int)fx - H + 1, b1 = (int)fy - H + 1, b2 = (int)fz - H + 1;
            const float tx = grid_frac(g.box, 0, p.x, fx), ty = grid_frac(g.box, 1, p.y, fy);
            if (lane < P) {
                const float d = (float)(lane - H + 1) - grid_frac(g.box, 2, p.z, fz);
                const float w = __expf(-d * d * g.hh[2]);
                zw[warp][lane] = make_float2(w, w * d * g.dfac[2]);
                zo[warp][lane] = (unsigned int)wrap_once(b2 + lane, n2) * plane;
            }
            // this lane's x points (weight 0 outside the stencil and for lanes past the last row)
            const int xs = (b0 & ~1) + 2 * slot;
            float wx[2], dx[2];
            #pragma unroll
            for (int v = 0; v < 2; ++v) {
                const int k = xs + v - b0;
                const float d = (float)(k - H + 1) - tx;
                wx[v] = k >= 0 && k < P && row < Sh::R ? __expf(-d * d * g.hh[0]) : 0.f;
                dx[v] = wx[v] * d * g.dfac[0];
            }
            const unsigned int xo = (unsigned int)wrap_once(xs, n0);
            unsigned int off[Sh::BL];
            float wy[Sh::BL], dy[Sh::BL];
            #pragma unroll
            for (int b = 0; b < Sh::BL; ++b) {
                const int j = row + Sh::R * b;
                const float d = (float)(j - H + 1) - ty;
                wy[b] = j < P ? __expf(-d * d * g.hh[1]) : 0.f;
                dy[b] = wy[b] * d * g.dfac[1];
                off[b] = (unsigned int)wrap_once(b1 + (j < P ? j : 0), n1) * (unsigned int)n0 + xo;
            }
            __syncwarp();
            float2 c0v[Sh::BL], c1v[Sh::BL];
            #pragma unroll
            for (int b = 0; b < Sh::BL; ++b) c0v[b] = c1v[b] = make_float2(0.f, 0.f);
            #pragma unroll
            for (int k = 0; k < P; ++k) {
                const float2 w = zw[warp][k];
                const unsigned int z = zo[warp][k];
                #pragma unroll
                for (int b = 0; b < Sh::BL; ++b) {
                    const float2 f = __ldg(reinterpret_cast<const float2*>(psi + (z + off[b])));
                    c0v[b] = __ffma2_rn(make_float2(w.x, w.x), f, c0v[b]);
                    c1v[b] = __ffma2_rn(make_float2(w.y, w.y), f, c1v[b]);
                }
            }
            float aphi = 0.f, ax = 0.f, ay = 0.f, az = 0.f;
            #pragma unroll
            for (int b = 0; b < Sh::BL; ++b) {
                const float r0 = fmaf(wx[1], c0v[b].y, wx[0] * c0v[b].x);
                const float r1 = fmaf(dx[1], c0v[b].y, dx[0] * c0v[b].x);
                const float r2 = fmaf(wx[1], c1v[b].y, wx[0] * c1v[b].x);
                aphi = fmaf(wy[b], r0, aphi);
                ax = fmaf(wy[b], r1, ax);
                ay = fmaf(dy[b], r0, ay);
                az = fmaf(wy[b], r2, az);
            }
            // reduce-scatter over the warp: lane 8 c ends with component c of (x, y, z, phi)
            const bool h4 = (lane & 16) != 0, h3 = (lane & 8) != 0;
            const float t0 = __shfl_xor_sync(0xffffffffu, h4 ? ax : az, 16);
            const float t1 = __shfl_xor_sync(0xffffffffu, h4 ? ay : aphi, 16);
            const float k0 = (h4 ? az : ax) + t0, k1 = (h4 ? aphi : ay) + t1;
            const float t2 = __shfl_xor_sync(0xffffffffu, h3 ? k0 : k1, 8);
            float v = (h3 ? k1 : k0) + t2;
            #pragma unroll
            for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((lane & 7) == 0)
                reinterpret_cast<float*>(far4 + s)[lane >> 3] = lane < 24 ? -p.w * v : v;
            __syncwarp();   // zw and zo are rewritten
        }
    }
    finish_psi_mean(ps, G, partial, counter, psi_mean);
}

/*
 * After the pair kernel and the far gather: per cluster slot t that holds an atom, the result in caller order,
 *   out[cperm[t]] = (F_near + F_far, phi_near + phi_far - F(0) q),
 * and the energies E = E_near + E_far + E_self (1/2 sum q phi over Eq. 20's near part, over the grid part,
 * and the self term -1/2 F(0) sum q^2), plus the net charge sum q (a diagnostic: the k = 0 term that a
 * non-zero net charge would carry is the one Eq. 4 drops).  Each block forms the four sums of its atoms;
 * the last block reduces them in block order.
 */
__global__ void __launch_bounds__(kThreads) k_combine(const float4* __restrict__ cpos,
                                                      const int* __restrict__ cperm,
                                                      const int* __restrict__ nslots,
                                                      const unsigned long long* __restrict__ near_acc,
                                                      const float4* __restrict__ far4, float F0, double F0d,
                                                      float wsum, const double* __restrict__ psi_mean,
                                                      float4* __restrict__ out, float4* __restrict__ near_dbg,
                                                      float4* __restrict__ far_dbg, double* __restrict__ partial,
                                                      unsigned int* __restrict__ counter,
                                                      double* __restrict__ energy,
                                                      double* __restrict__ net_charge, int max_atoms,
                                                      int max_slots, int* __restrict__ status)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    __shared__ double red[kWarps][4];
    __shared__ int is_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float phi_dc = (float)(*psi_mean) * wsum;   // potential of psi's rounding-level k = 0 mode
    CSum qn, qf, qq, qs;                              // sums of q phi_near, q phi_far, q^2, q
    const int ns = *nslots;
    for (int t = blockIdx.x * kThreads + threadIdx.x; t < ns; t += gridDim.x * kThreads) {
        if (!USR_IN_BOUNDS(t, max_slots, status)) continue;
        const int i = cperm[t];
        const float4 nr = near_part(near_acc, t), f = far4[t];
        const float qi = cpos[t].w;
        if (i < 0) continue;                          // a padding slot
        const float phi_far = f.w - phi_dc;
        qn.add_product(qi, nr.w);
        qf.add_product(qi, phi_far);
        qq.add_product(qi, qi);
        qs.add(qi);
        if (!USR_IN_BOUNDS(i, max_atoms, status)) continue;
        out[i] = make_float4(nr.x + f.x, nr.y + f.y, nr.z + f.z, nr.w + phi_far - F0 * qi);
        if (near_dbg) near_dbg[i] = nr;
        if (far_dbg) far_dbg[i] = make_float4(f.x, f.y, f.z, phi_far);
    }
    double e[4] = {0.5 * warp_sum_c(qn), 0.5 * warp_sum_c(qf), -0.5 * F0d * warp_sum_c(qq), warp_sum_c(qs)};
    if (lane == 0)
        for (int c = 0; c < 4; ++c) red[warp][c] = e[c];
    __syncthreads();
    if (threadIdx.x < 4) {
        double v = 0.0;
        for (int w = 0; w < kWarps; ++w) v += red[w][threadIdx.x];
        partial[(size_t)blockIdx.x * 4 + threadIdx.x] = v;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!is_last) return;
    // the last CTA: the four sums over all CTAs in a fixed order
    __threadfence();
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = threadIdx.x; k < (int)gridDim.x; k += kThreads)
        for (int c = 0; c < 4; ++c) acc[c] += ((volatile double*)partial)[(size_t)k * 4 + c];
    for (int c = 0; c < 4; ++c) acc[c] = warp_sum_d(acc[c]);
    __syncthreads();
    if (lane == 0)
        for (int c = 0; c < 4; ++c) red[warp][c] = acc[c];
    __syncthreads();
    if (threadIdx.x == 0) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int w = 0; w < kWarps; ++w)
            for (int c = 0; c < 4; ++c) v[c] += red[w][c];
        energy[0] = v[0] + v[1] + v[2];
        energy[1] = v[0];
        energy[2] = v[1];
        energy[3] = v[2];
        *net_charge = v[3];
        *counter = 0u;
    }
}

/* ------------------------------------------------------------------ launch */

#define USR_GATHER_CASE(PP)                                                                                          \
    case PP:                                                                                                         \
        launch_with(-1, k_gather<PP>, nb, kGThreads, 0, st, L.cpos, L.pstart + ncell, psi, g, far4, partial,         \
                    counter, psi_mean, status);                                                                      \
        break;

/* Cluster slots of n atoms in ncell cells at most. */
static int max_slots_of(int n, int ncell)
{
    return (int)std::min((long long)n + 7LL * std::min(n, ncell), (long long)INT_MAX);
}

static int gather_blocks(int n, int P)
{
    const int apc = kGThreads / gather_lanes(P);   // atoms per CTA pass
    return std::max(1, std::min(kGatherBlocks, (n + apc - 1) / apc));
}

template <int P>
static void gather_wide(int n, const ClusterList& L, int ncell, const float* psi, const GridArgs& g, float4* far4,
                        double* partial, unsigned int* counter, double* psi_mean, int* status, cudaStream_t st)
{
    // slots per warp and pass: up to 8 neighbours (their rows overlap in L1), fewer when that would leave warps idle
    const int slots = max_slots_of(n, ncell), per = std::max(1, std::min(8, slots / (kGWarps * kGatherBlocks)));
    const int nb = std::max(1, std::min(kGatherBlocks, (slots + kGWarps * per - 1) / (kGWarps * per)));
    launch_with(-1, k_gather_wide<P>, nb, kGThreads, 0, st, L.cpos, L.pstart + ncell, per, psi, g, far4, partial,
                counter, psi_mean, status);
}

void launch_gather(int P, int n, const ClusterList& L, int ncell, const float* psi, const GridArgs& g, float4* far4,
                   double* partial, unsigned int* counter, double* psi_mean, int* status, cudaStream_t st)
{
    const int nb = gather_blocks(max_slots_of(n, ncell), P);
    if (P >= 12 && g.box.n[0] % 2 == 0) {
        if (P == 12) gather_wide<12>(n, L, ncell, psi, g, far4, partial, counter, psi_mean, status, st);
        else if (P == 14) gather_wide<14>(n, L, ncell, psi, g, far4, partial, counter, psi_mean, status, st);
        else gather_wide<16>(n, L, ncell, psi, g, far4, partial, counter, psi_mean, status, st);
        return;
    }
    switch (P) {
        USR_GATHER_CASE(8)
        USR_GATHER_CASE(10)
        USR_GATHER_CASE(12)
        USR_GATHER_CASE(14)
        default:
        USR_GATHER_CASE(16)
    }
}

void launch_combine(int n, const ClusterList& L, int ncell, const unsigned long long* near_acc, const float4* far4,
                    const GridArgs& g, float4* out, float4* near_dbg, float4* far_dbg, double* partial,
                    unsigned int* counter, double* energy, double* net_charge, int* status, cudaStream_t st)
{
    const int nb = std::max(1, std::min(kCombineBlocks, (max_slots_of(n, ncell) + kThreads - 1) / kThreads));
    k_combine<<<nb, kThreads, 0, st>>>(L.cpos, L.cperm, L.pstart + ncell, near_acc, far4, g.F0, g.F0d, g.wsum,
                                       g.psi_mean, out, near_dbg, far_dbg, partial, counter, energy, net_charge, n,
                                       g.max_slots, status);
}

}  // namespace usr

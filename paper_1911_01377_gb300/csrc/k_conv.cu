/*
 * k_conv.cu -- the separable real-space far-part convolutions (Sec. V,
 * Eqs. 31-32): for each Gaussian term j < N the on-grid potential is the
 * composition of three 1D circular convolutions, and the N results are
 * summed.  Each 1D pass contracts one grid axis with an n x n circulant
 * matrix, so each pass is a (batched) GEMM:
 *
 *   x pass  X_j[z][y][:] = rho[z][y][:] . K_j^x       all terms in one GEMM,
 *           M = ny nz lines, N = N_terms nx, K = nx (the terms share the rho read)
 *   y pass  Y_j[z] = K_j^y . X_j[z]                  batched over (j, z)
 *   z pass  psi = sum_j scale_j K_j^z . Y_j           one GEMM, K = N_terms nz,
 *           the sum over terms is part of the contraction
 *
 * Every 1D kernel is stored as its zero-mean part K~ (circulant) plus its
 * mean mu: K v = K~ v + mu (sum v).  Wide Gaussians are almost constant on
 * the period, so rounding K itself to FP32 would bury their small non-constant
 * part; the split keeps it at full FP32 relative accuracy.  The DC term is the
 * GEMM's rank-one epilogue: row sums of A (x pass, which also subtracts the
 * grid mean: the dropped k = 0 mode) or weighted column sums of B (y, z).
 *
 * This is the plain FP32 CUDA-core form: tiles of TM x TN outputs by 16 of K in shared memory, two of them (the next
 * one's global loads are in flight while this one is multiplied), 128 threads, TM / 8 x TN / 16 outputs each.  Every
 * 16 products are summed apart and then added to the output (shorter rounding chains for K up to terms x n).
 *
 * Bound: latency.  A pass has 30 to 400 tiles of 64 x 64 and 2 to 25 steps along K; without the second buffer every
 * step waited for its loads (slab 64 x 64 x 80, 5 terms: 18, 19 and 45 us alone for the three passes).  The tile
 * shrinks to 32 x 64 and 32 x 32 when larger ones would leave SMs idle.
 */
#include "usr_internal.h"

namespace usr {

namespace {
constexpr int BK = 16, kThreads = 128;

/* W consecutive floats of p from index i on, zero from `end` on; one wide load per four when vec and all inside. */
template <int W>
__device__ __forceinline__ void load_run(float (&v)[W], const float* __restrict__ p, int i, int end, bool vec)
{
    #pragma unroll
    for (int q = 0; q < W; q += 4) {
        if (vec && i + q + 3 < end) {
            const float4 f = __ldg(reinterpret_cast<const float4*>(p + i + q));
            v[q] = f.x;
            v[q + 1] = f.y;
            v[q + 2] = f.z;
            v[q + 3] = f.w;
        } else {
            #pragma unroll
            for (int c = 0; c < 4; ++c) v[q + c] = i + q + c < end ? __ldg(p + i + q + c) : 0.f;
        }
    }
}
}  // namespace

/* vec: the rows of A and B start on 16-byte boundaries. */
template <int TM, int TN, int MODE>
__global__ void __launch_bounds__(kThreads) k_conv_gemm(ConvGemm g, int vec)
{
    pdl_wait();   // the predecessor on this stream has completed (programmatic launch)
    constexpr int RM = TM / 8, RN = TN / 16;           // outputs per thread
    constexpr int WA = TM * BK / kThreads, WB = TN * BK / kThreads;   // floats of A and B a thread stages
    __shared__ __align__(16) float As[2][BK][TM + 4];
    __shared__ __align__(16) float Bs[2][BK][TN + 4];
    __shared__ float dc[64];
    const int batch = blockIdx.z;
    const int b1 = batch / g.nb2, b2 = batch - b1 * g.nb2;
    const float* __restrict__ A = g.A + b1 * g.a_s1 + b2 * g.a_s2;
    const float* __restrict__ B = g.B + b1 * g.b_s1 + b2 * g.b_s2;
    const float* __restrict__ w = g.dcw ? g.dcw + b1 * g.dcw_s1 : nullptr;
    const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int M = g.M, N = g.N, K = g.K;
    const int ar = tid / (BK / WA), ak = tid % (BK / WA) * WA;       // A: row and first k of this thread's run
    const int bk = tid / (TN / WB), bc = tid % (TN / WB) * WB;       // B: k and first column
    float ra[WA], rb[WB], acc[RM][RN];
    #pragma unroll
    for (int i = 0; i < RM; ++i)
        #pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = 0.f;
    float dcacc = 0.f;
    auto fetch = [&](int k0) {
        load_run<WA>(ra, A + (long long)(m0 + ar) * g.lda, k0 + ak, m0 + ar < M ? K : 0, vec != 0);
        load_run<WB>(rb, B + (long long)(k0 + bk) * g.ldb, n0 + bc, k0 + bk < K ? N : 0, vec != 0);
    };
    auto stage = [&](int s) {
        #pragma unroll
        for (int q = 0; q < WA; ++q) As[s][ak + q][ar] = ra[q];
        #pragma unroll
        for (int q = 0; q < WB; q += 4)
            *reinterpret_cast<float4*>(&Bs[s][bk][bc + q]) = make_float4(rb[q], rb[q + 1], rb[q + 2], rb[q + 3]);
    };
    fetch(0);
    stage(0);
    __syncthreads();
    for (int k0 = 0, s = 0; k0 < K; k0 += BK, s ^= 1) {
        const bool more = k0 + BK < K;
        if (more) fetch(k0 + BK);
        if (MODE == 1 && tid < TM) {
            float t = 0.f;
            #pragma unroll
            for (int kk = 0; kk < BK; ++kk) t += As[s][kk][tid];
            dcacc += t;
        }
        if (MODE == 2 && tid < TN) {
            float t = 0.f;
            #pragma unroll
            for (int kk = 0; kk < BK; ++kk)
                if (k0 + kk < K) t = fmaf(__ldg(&w[k0 + kk]), Bs[s][kk][tid], t);
            dcacc += t;
        }
        float c[RM][RN];
        #pragma unroll
        for (int i = 0; i < RM; ++i)
            #pragma unroll
            for (int j = 0; j < RN; ++j) c[i][j] = 0.f;
        #pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[RM], b[RN];
            #pragma unroll
            for (int i = 0; i < RM; i += 4) {
                const float4 f = *reinterpret_cast<const float4*>(&As[s][kk][ty * RM + i]);
                a[i] = f.x;
                a[i + 1] = f.y;
                a[i + 2] = f.z;
                a[i + 3] = f.w;
            }
            #pragma unroll
            for (int j = 0; j < RN; j += 2) {
                const float2 f = *reinterpret_cast<const float2*>(&Bs[s][kk][tx * RN + j]);
                b[j] = f.x;
                b[j + 1] = f.y;
            }
            #pragma unroll
            for (int i = 0; i < RM; ++i)
                #pragma unroll
                for (int j = 0; j < RN; ++j) c[i][j] = fmaf(a[i], b[j], c[i][j]);
        }
        #pragma unroll
        for (int i = 0; i < RM; ++i)
            #pragma unroll
            for (int j = 0; j < RN; ++j) acc[i][j] += c[i][j];
        if (more) stage(s ^ 1);       // the other buffer: its readers passed the barrier of the step before
        __syncthreads();
    }
    if (MODE != 0) {
        if (tid < (MODE == 1 ? TM : TN)) {
            float v = dcacc;
            if (MODE == 1 && g.mean) v -= (float)((double)K * *g.mean);
            dc[tid] = v;
        }
        __syncthreads();
    }
    float* __restrict__ C = g.C + b1 * g.c_s1 + b2 * g.c_s2;
    #pragma unroll
    for (int i = 0; i < RM; ++i) {
        const int m = m0 + ty * RM + i;
        if (m >= M) continue;
        #pragma unroll
        for (int j = 0; j < RN; ++j) {
            const int n = n0 + tx * RN + j;
            if (n >= N) continue;
            float v = acc[i][j];
            if (MODE == 1) v = fmaf(__ldg(&w[n]), dc[ty * RM + i], v);
            if (MODE == 2) v += dc[tx * RN + j];
            const int jb = n / g.nsplit;
            const int nn = n - jb * g.nsplit;
            C[jb * g.c_split + (long long)m * g.ldc + nn] = v;
        }
    }
}

template <int TM, int TN>
static void launch_tile(const ConvGemm& g, int batches, int vec, cudaStream_t st)
{
    const dim3 grid((g.N + TN - 1) / TN, (g.M + TM - 1) / TM, batches);
    switch (g.mode) {
        case 1: launch_pdl(k_conv_gemm<TM, TN, 1>, grid, kThreads, 0, st, g, vec); break;
        case 2: launch_pdl(k_conv_gemm<TM, TN, 2>, grid, kThreads, 0, st, g, vec); break;
        default: launch_pdl(k_conv_gemm<TM, TN, 0>, grid, kThreads, 0, st, g, vec); break;
    }
}

/* The largest tile that still gives every SM two CTAs (measured on the slab's z pass, M = 80, N = 4096, K = 400: 64 x 64
   wastes 3/8 of its second row of tiles and has 128 CTAs). */
void launch_conv(const ConvGemm& g, int batches, cudaStream_t st)
{
    auto row16 = [](const float* p, long long ld, long long s1, long long s2) {
        return ((uintptr_t)p & 15) == 0 && ld % 4 == 0 && s1 % 4 == 0 && s2 % 4 == 0;
    };
    const int vec = row16(g.A, g.lda, g.a_s1, g.a_s2) && row16(g.B, g.ldb, g.b_s1, g.b_s2);
    auto ctas = [&](int tm, int tn) { return (long long)((g.M + tm - 1) / tm) * ((g.N + tn - 1) / tn) * batches; };
    if (ctas(64, 64) >= 304)
        launch_tile<64, 64>(g, batches, vec, st);
    else if (ctas(32, 64) >= 304)
        launch_tile<32, 64>(g, batches, vec, st);
    else
        launch_tile<32, 32>(g, batches, vec, st);
}

}  // namespace usr

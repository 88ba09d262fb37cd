// Adjoint of the Lenia step with global genes (no gene maps, no alpha):
//   U_k  = K~_k * A_src(k)
//   g_k  = exp(-(U_k - mu_k)^2 / (2 sigma_k^2)),  F(g) = 2g - 1 (signed) or g (paper form)
//   pre_c = A_c + dt sum_{k: dst(k)=c} h_k F(g_k),   A'_c = clip(pre_c, 0, 1)
// Given dL/dA' this computes, per site,
//   gpre_c = dL/dA'_c [0 < pre_c < 1]                (clip subgradient)
//   gU_k   = gpre_dst(k) dt h_k F'(g) g (-(U - mu) / sigma^2)
// and the per-kernel gene gradients
//   dL/dmu_k    = sum gpre dt h_k F' g (U - mu) / sigma^2
//   dL/dsigma_k = sum gpre dt h_k F' g (U - mu)^2 / sigma^3
//   dL/dh_k     = sum gpre dt F(g)
// as block partials in compensated FP32 pairs (hi + lo) that every reversed step
// adds to, reduced once per pass in a fixed order (one block per value).  The
// transposed convolution (gA_src += K~_k (x) gU_k; K~ is point symmetric, so
// it is the same convolution) runs on the forward machinery; its inverse pass
// adds gpre, or - where every gradient plane is convolved by itself - the next
// reversed step gathers gpre + sum_k V_k as it reads.
#include "lenia_internal.cuh"
#include "ptx_util.cuh"

namespace lenia {

constexpr int ADJ_THREADS = 128;
constexpr int ADJ_KB = 16;              // kernels whose gene terms meet in shared memory at a time
constexpr float ADJ_HALF_LOG2E = 0.721347520444481703680f;   // 0.5 log2(e)

// One site per thread; the growth is recomputed with the same arithmetic as
// the forward streaming epilogue so that clip decisions match.  A site's bumps
// and channel sums sit in its thread's column of shared memory (kernel counts
// and routing are run-time values), and the gene terms of ADJ_KB kernels at a
// time are summed over the block from there in compensated pairs, four values a
// warp (256^2, 15 kernels: 17 -> 8 us with the gather; a pass of 12 steps 1.05 ms
// with a shuffle tree of pairs per value).
__global__ void __launch_bounds__(ADJ_THREADS) k_adjoint_epilogue(const __grid_constant__ AdjParams p)
{
    pdl_enter();
    extern __shared__ float adj_sm[];
    const int K = p.kt.K, C = p.kt.C, tid = threadIdx.x;
    float* bump = adj_sm;                                   // [K][T]
    float* chan = bump + (size_t)K * ADJ_THREADS;           // [C][T]: pre-clip sum, then gpre
    float* inc = chan + (size_t)C * ADJ_THREADS;            // [C][T]: dL/dA_{t+1}
    float* red = inc + (size_t)C * ADJ_THREADS;             // [3 ADJ_KB][T]
    const size_t N = (size_t)p.H * p.W;
    const size_t i = (size_t)blockIdx.x * ADJ_THREADS + tid;
    const bool valid = i < N;
    const size_t ic = valid ? i : N - 1;
    const int lane = tid & 31, warp = tid >> 5;

    for (int c = 0; c < C; c++) {
        chan[c * ADJ_THREADS + tid] = 0.f;
        inc[c * ADJ_THREADS + tid] = p.gpre_prev ? 0.f : __ldg(p.gA_next + (size_t)c * N + ic);
    }
    if (p.gpre_prev) {
        // the planes among themselves first: they are small beside gpre (dt), and a
        // sum that starts from gpre rounds at its size once per kernel (256^2, 15
        // kernels: 1.9e-7 of dL/dA_0 against 1.4e-7)
#pragma unroll 5
        for (int k = 0; k < K; k++) inc[p.kt.src[k] * ADJ_THREADS + tid] += __ldg(&p.V[(size_t)k * N + ic]);
        for (int c = 0; c < C; c++) inc[c * ADJ_THREADS + tid] += __ldg(p.gpre_prev + (size_t)c * N + ic);
    }
#pragma unroll 5
    for (int k = 0; k < K; k++) {
        const float u = __ldg(&p.U[(size_t)k * N + ic]);
        const float z = (u - p.kt.mu[k]) * rcp_approx(p.kt.sigma[k]);
        const float g = ex2_approx(-ADJ_HALF_LOG2E * (z * z));
        const float h = p.kt.h[k];
        bump[k * ADJ_THREADS + tid] = g;
        chan[p.kt.dst[k] * ADJ_THREADS + tid] += p.growth_form == 0 ? fmaf(2.f * g, h, -h) : h * g;
    }
    for (int c = 0; c < C; c++) {
        const float a = __ldg(&p.A[(size_t)c * N + ic]) + p.dt * chan[c * ADJ_THREADS + tid];
        const float gpre = valid && a > 0.f && a < 1.f ? inc[c * ADJ_THREADS + tid] : 0.f;
        chan[c * ADJ_THREADS + tid] = gpre;
        if (valid) p.gpre[(size_t)c * N + i] = gpre;
    }
    // kernel by kernel: potential gradient and this block's gene partials
    const float fp = p.growth_form == 0 ? 2.f : 1.f;        // F'(g)
    for (int k0 = 0; k0 < K; k0 += ADJ_KB) {
        const int kn = min(ADJ_KB, K - k0);
#pragma unroll 3
        for (int j = 0; j < kn; j++) {
            const int k = k0 + j;
            const float d = __ldg(&p.U[(size_t)k * N + ic]) - p.kt.mu[k];
            const float h = p.kt.h[k];
            const float g = bump[k * ADJ_THREADS + tid];
            const float gp = chan[p.kt.dst[k] * ADJ_THREADS + tid] * p.dt;
            const float w = gp * h * fp * g;                // dL/d(exp term)
            const float wd = w * d * p.inv_s2[k];
            if (valid) p.gU[(size_t)k * N + i] = -wd;
            red[(3 * j) * ADJ_THREADS + tid] = wd;
            red[(3 * j + 1) * ADJ_THREADS + tid] = wd * d;
            red[(3 * j + 2) * ADJ_THREADS + tid] = gp * (p.growth_form == 0 ? 2.f * g - 1.f : g);
        }
        __syncthreads();
        // value-major partials [K * 3][blocks]: the reduction kernel reads them coalesced.
        // Four values a warp: the lanes halve twice over the values, then three times
        // over the sites, and lanes 0, 8, 16 and 24 end with a value each.
        for (int v0 = 4 * warp; v0 < 3 * kn; v0 += ADJ_THREADS / 8) {
            float2 t[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const float* r = red + min(v0 + j, 3 * kn - 1) * ADJ_THREADS + lane;
                t[j] = ff_add(ff_add(make_float2(r[0], 0.f), make_float2(r[32], 0.f)),
                              ff_add(make_float2(r[64], 0.f), make_float2(r[96], 0.f)));
            }
            const bool hi = lane & 16, mid = lane & 8;
            const float2 s0 = ff_shfl_xor(hi ? t[0] : t[2], 16), s1 = ff_shfl_xor(hi ? t[1] : t[3], 16);
            const float2 h0 = ff_add(hi ? t[2] : t[0], s0), h1 = ff_add(hi ? t[3] : t[1], s1);
            float2 u = ff_add(mid ? h1 : h0, ff_shfl_xor(mid ? h0 : h1, 8));
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) u = ff_add(u, ff_shfl_xor(u, off));
            const int v = v0 + (hi ? 2 : 0) + (mid ? 1 : 0);
            if ((lane & 7) == 0 && v < 3 * kn) {
                if (v % 3 == 1) {
                    // dL/dsigma: the sum's sites share the division by sigma
                    const float sg = p.kt.sigma[k0 + v / 3], q = u.x / sg;
                    u = make_float2(q, (fmaf(-q, sg, u.x) + u.y) / sg);
                }
                float2* o = p.gene_partials + (size_t)(3 * k0 + v) * gridDim.x + blockIdx.x;
                *o = p.first ? u : ff_add(*o, u);
            }
        }
        __syncthreads();
    }
}

// gene_acc[v] = sum over the nb block partials of value v (block v): thread t
// sums blocks t, t + 256, ... in order, then a fixed shuffle / shared tree,
// so every launch adds in the same order.
constexpr int ADJ_RED_THREADS = 256;
__global__ void __launch_bounds__(ADJ_RED_THREADS) k_adjoint_gene_reduce(const float2* partials, int nb,
                                                                      float2* gene_acc)
{
    pdl_enter();
    __shared__ float2 wsum[ADJ_RED_THREADS / 32];
    const int v = blockIdx.x;
    const float2* src = partials + (size_t)v * nb;
    float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
    int b = threadIdx.x;
    for (; b + ADJ_RED_THREADS < nb; b += 2 * ADJ_RED_THREADS) {
        s0 = ff_add(s0, src[b]);
        s1 = ff_add(s1, src[b + ADJ_RED_THREADS]);
    }
    if (b < nb) s0 = ff_add(s0, src[b]);
    float2 s = ff_add(s0, s1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s = ff_add(s, ff_shfl_down(s, off));
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float2 t = make_float2(0.f, 0.f);
        for (int w = 0; w < ADJ_RED_THREADS / 32; w++) t = ff_add(t, wsum[w]);
        gene_acc[v] = t;
    }
}

// gA_c = gpre_c + sum_{k: src(k) = c} V_k  (V_k = K~_k (x) gU_k, in kernel order),
// or gpre_c + V_c when the sum over kernels was taken in the frequency domain
__global__ void __launch_bounds__(256) k_adjoint_gather(AdjParams p)
{
    pdl_enter();
    const size_t N = (size_t)p.H * p.W;
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= N) return;
    for (int c = 0; c < p.kt.C; c++) {
        float s = __ldg(&p.gpre[(size_t)c * N + i]);
        if (p.v_per_channel) {
            s += __ldg(&p.V[(size_t)c * N + i]);
        } else {
            for (int k = 0; k < p.kt.K; k++)
                if (p.kt.src[k] == c) s += __ldg(&p.V[(size_t)k * N + i]);
        }
        p.gA_out[(size_t)c * N + i] = s;
    }
}

__global__ void k_adjoint_gene_out(const float2* gene_acc, int nv, float* out)
{
    pdl_enter();
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < nv) out[v] = gene_acc[v].x + gene_acc[v].y;
}

int adjoint_blocks(int H, int W) { return (int)(((size_t)H * W + ADJ_THREADS - 1) / ADJ_THREADS); }

cudaError_t launch_adjoint_epilogue(const AdjParams& p0, cudaStream_t s)
{
    AdjParams p = p0;
    for (int k = 0; k < p.kt.K; k++) p.inv_s2[k] = (float)(1.0 / ((double)p.kt.sigma[k] * p.kt.sigma[k]));
    const size_t smem = (size_t)(p.kt.K + 2 * p.kt.C + 3 * ADJ_KB) * ADJ_THREADS * sizeof(float);
    // one limit for every kernel count: threads with different worlds may come here at once
    constexpr size_t most = (size_t)(kMaxKernels + 2 * kMaxChannels + 3 * ADJ_KB) * ADJ_THREADS * sizeof(float);
    cudaError_t e = smem_limit<k_adjoint_epilogue>(most);
    if (e != cudaSuccess) return e;
    launch_pdl(k_adjoint_epilogue, adjoint_blocks(p.H, p.W), ADJ_THREADS, smem, s, p);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_gene_reduce(const float2* partials, int H, int W, int nv, float2* gene_acc, cudaStream_t s)
{
    launch_pdl(k_adjoint_gene_reduce, nv, ADJ_RED_THREADS, 0, s, partials, adjoint_blocks(H, W), gene_acc);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_gather(const AdjParams& p, cudaStream_t s)
{
    const size_t N = (size_t)p.H * p.W;
    launch_pdl(k_adjoint_gather, (unsigned)((N + 255) / 256), 256, 0, s, p);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_gene_out(const float2* gene_acc, int nv, float* out, cudaStream_t s)
{
    launch_pdl(k_adjoint_gene_out, (nv + 63) / 64, 64, 0, s, gene_acc, nv, out);
    return cudaGetLastError();
}

}  // namespace lenia

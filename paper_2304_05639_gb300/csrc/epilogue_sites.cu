// The per-site rule after the convolution (diffusion, growth, alpha, masking,
// clipped update; arXiv 2304.05639, Sections 2.1-2.4, Algorithm 2) for any
// kernel count, channel count and growth-gene layout, and diffusion radius 1 or 2.
//
// A thread takes four adjacent columns of one row and walks the kernels: each
// gene plane's stencil comes in as float4 rows plus the two or four neighbours to
// the left and right, the kernel's genes are diffused, its growth added to
// its channel, and the diffused genes go straight back out (zeros once alpha is
// known to be false; sites that turn out false later rewrite theirs).  A
// block covers 32 columns x 16 rows at a time and strides over the world.
//
// Where the genes are maintained, a site whose disk holds no first gene above
// eps_p has alpha = 0 whatever the rest says: its genes are zero and its update
// is the per-channel constant.  A warp (32 columns x 4 rows) of such sites (the
// empty part of a world, most of it in the worlds of the paper) reads one gene
// plane instead of all of them and no potential.
//
// The arithmetic is the hardware reciprocal (with one correction for the genes)
// and exponential.  Alpha tests that its rounding, or the rounding of the
// windows' potentials, could turn count as passed until the kernels are done; the
// sites that hang on them are then dealt to the warp's lanes and settled by the
// other update kernels' arithmetic on the direct sums, so that a world's
// decisions do not depend on the kernel or the convolution it takes.  (Settled
// inside the kernels' loop, or with a site of each lane at a time, the guard that
// large radii need makes a step of 600 x 900 at R = 45 / 56 1.15 / 2.25 ms; 0.22 /
// 0.62 so, 0.56 / 0.93 with the direct sums throughout.)
//
// What bounds it: on a mostly empty world the writes of the gene planes, on a
// full one its loads and instruction issue (16 warps an SM at 128 registers, half of
// the issue slots used).  1080 x 1920, 15 kernels, 43% live: 128 us on cold caches
// (533 with the general kernel; 146 with every lane loading its own stencils), of
// which settling takes 5; 512^2, 8 kernels, three genes, radius 2: 24 us (230).
#include <math.h>
#include <string.h>

#include "lenia_internal.cuh"
#include "ptx_util.cuh"

namespace lenia {
namespace {

constexpr int ES_Q = 8, ES_Y = 16;                 // quads and rows of a block (128 threads)
constexpr int ES_T = ES_Q * ES_Y, ES_NW = ES_T / 32;

struct SitesParams {
    EpiParams e;
    int n_worlds;              // worlds of a batched launch (lists in e), else 1
    int tx, ty;                // blocks of 32 x 16 sites per world
    int gate;
    int tiny_eps;              // the threshold lies where bumps underflow
    int fast;                  // settle with reciprocals and the hardware exponential, else divisions and expf
    GuardParams g;
};

// One gene plane around a quad: rows y - RD .. y + RD, columns x - RD .. x + 3 + RD.
template <int RD>
struct Stencil {
    float v[2 * RD + 1][4 + 2 * RD];
    __device__ __forceinline__ static constexpr int half(int dy)
    {
        return RD == 0 ? 0 : RD == 1 ? (dy == 0 ? 1 : 0) : (dy == 0 ? 2 : (dy == 2 || dy == -2) ? 0 : 1);
    }
    // pl: the plane at the quad; ro[]: row offsets from y; xl[], xr[]: offsets of the
    // columns to the left and right; c: the quad itself
    __device__ __forceinline__ void load(const float* pl, const int* ro, const int* xl, const int* xr, float4 c)
    {
#pragma unroll
        for (int j = 0; j <= 2 * RD; j++) {
            const float* row = pl + ro[j];
            const float4 f = j == RD ? c : __ldg(reinterpret_cast<const float4*>(row));
            v[j][RD] = f.x;
            v[j][RD + 1] = f.y;
            v[j][RD + 2] = f.z;
            v[j][RD + 3] = f.w;
#pragma unroll
            for (int i = 1; i <= RD; i++)
                if (i <= half(j - RD)) {
                    v[j][RD - i] = __ldg(row + xl[i - 1]);
                    v[j][RD + 3 + i] = __ldg(row + xr[i - 1]);
                }
        }
    }
    __device__ __forceinline__ bool any_above(float eps) const
    {
        float m = v[RD][RD];
#pragma unroll
        for (int j = 0; j <= 2 * RD; j++)
#pragma unroll
            for (int i = 0; i < 4 + 2 * RD; i++)
                if (i >= RD - half(j - RD) && i < 4 + RD + half(j - RD)) m = fmaxf(m, v[j][i]);
        return m > eps;
    }
    // P^ of the four columns: the disk's sum (rows, then columns) over the count above eps_p, clipped
    __device__ __forceinline__ void diffused(float eps, float* out) const
    {
        float one[2 * RD + 1][4 + 2 * RD];
#pragma unroll
        for (int j = 0; j <= 2 * RD; j++)
#pragma unroll
            for (int i = 0; i < 4 + 2 * RD; i++)
                if (i >= RD - half(j - RD) && i < 4 + RD + half(j - RD)) one[j][i] = v[j][i] > eps ? 1.f : 0.f;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            float s = 0.f, n = 0.f;
#pragma unroll
            for (int j = 0; j <= 2 * RD; j++)
#pragma unroll
                for (int d = -RD; d <= RD; d++)
                    if (d <= half(j - RD) && -d <= half(j - RD)) {
                        const bool first = j == 0;
                        s = first ? v[j][RD + c + d] : s + v[j][RD + c + d];
                        n = first ? one[j][RD + c + d] : n + one[j][RD + c + d];
                    }
            // (2 stands for a larger quotient: an infinite one's correction would be infinity
            // less infinity, and it saturates to 1 all the same)
            const float rn = rcp_approx(n), t = fminf(s * rn, 2.f);
            const float r = fmaf(fmaf(-t, n, s), rn, t);
            out[c] = n > 0.f ? __saturatef(r) : 0.f;
        }
    }
};

// Tap t of the list: its value's place in the plane, and its weight.
__device__ __forceinline__ int tap_site(int2 tap, int y, int x, int H, int W)
{
    int yy = y + (tap.x >> 11) - 1024, xx = x + (tap.x & 2047) - 1024;
    yy = yy < 0 ? yy + H : (yy >= H ? yy - H : yy);
    xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
    return yy * W + xx;
}

// Kernel k's direct sum at (y, x): its non-zero taps in k_direct_conv's order (a zero
// weight adds nothing there), so the same bits.  By a whole warp: the lanes fetch 128
// taps at once, the next ones while every lane adds these, in order, from shared
// memory (sm: the warp's).  At usual radii a step has a few such sites and they cost
// its latency: 436 taps of R = 12 took 14000 cycles with the operands passed round
// by shuffles, 10000 with the taps fetched just before their values (six steps of
// 300 x 404 120, 109 and 94 us).
constexpr int ES_TAPS = 128;
__device__ __forceinline__ float direct_warp(const SitesParams& q, const float* A, int k, int y, int x, float2* sm)
{
    constexpr int B = ES_TAPS / 32;
    const int H = q.e.H, W = q.e.W, lane = threadIdx.x & 31;
    const float* plane = A + (size_t)q.e.kt.src[k] * H * W;
    const int t1 = q.g.off[k + 1];
    // taps a batch ahead of their values, values a batch ahead of their sums
    int2 tap[B];
    float2 next[B];
    auto fetch_taps = [&](int t0) {
#pragma unroll
        for (int j = 0; j < B; j++) {
            const int t = t0 + 32 * j + lane;
            tap[j] = t < t1 ? __ldg(&q.g.taps[t]) : make_int2((1024 << 11) + 1024, 0);
        }
    };
    auto fetch_values = [&]() {                // (beyond t1: the site itself by 0)
#pragma unroll
        for (int j = 0; j < B; j++)
            next[j] = make_float2(__int_as_float(tap[j].y), __ldg(&plane[tap_site(tap[j], y, x, H, W)]));
    };
    float acc = 0.f;
    fetch_taps(q.g.off[k]);
    fetch_values();
    fetch_taps(q.g.off[k] + ES_TAPS);
#pragma unroll 1
    for (int t0 = q.g.off[k]; t0 < t1; t0 += ES_TAPS) {
#pragma unroll
        for (int j = 0; j < B; j++) sm[32 * j + lane] = next[j];
        __syncwarp();
        fetch_values();
        fetch_taps(t0 + 2 * ES_TAPS);
        const float2* e = sm;
        const int n = min(ES_TAPS, t1 - t0);
        int i = 0;
#pragma unroll 1
        for (; i + 16 <= n; i += 16) {
            float4 f[8];
#pragma unroll
            for (int j = 0; j < 8; j++) f[j] = reinterpret_cast<const float4*>(e + i)[j];
#pragma unroll
            for (int j = 0; j < 8; j++) acc = fmaf(f[j].z, f[j].w, fmaf(f[j].x, f[j].y, acc));
        }
#pragma unroll 1
        for (; i < n; i++) acc = fmaf(e[i].x, e[i].y, acc);
        __syncwarp();
    }
    return acc;
}

// The direct sums of the lanes that want one (the whole warp calls it).  Up to four
// sites take the warp one after the other; more go side by side, a lane each
// (a sum's additions are one chain), the taps read from shared memory.
__device__ __forceinline__ float direct_sums(const SitesParams& q, const float* A, int k, int y, int x, bool want, float2* sm)
{
    constexpr int B = 8;
    const int H = q.e.H, W = q.e.W, lane = threadIdx.x & 31, R = q.g.R;
    uint32_t m = __ballot_sync(0xffffffffu, want);
    const int t1 = q.g.off[k + 1];
    float acc = 0.f;
    if (__popc(m) <= 4) {
#pragma unroll 1
        for (; m; m &= m - 1) {
            const int L = __ffs(m) - 1;
            const float s = direct_warp(q, A, k, __shfl_sync(0xffffffffu, y, L), __shfl_sync(0xffffffffu, x, L), sm);
            if (lane == L) acc = s;
        }
        return acc;
    }
    // the other lanes read along at the first site
    const int L = __ffs(m) - 1, y0 = __shfl_sync(0xffffffffu, y, L), x0 = __shfl_sync(0xffffffffu, x, L);
    if (!want) {
        y = y0;
        x = x0;
    }
    const bool inner = __all_sync(0xffffffffu, y >= R && y < H - R && x >= R && x < W - R);
    const float* plane = A + (size_t)q.e.kt.src[k] * H * W;
    const float* at = plane + (size_t)y * W + x;
    int2 next = make_int2((1024 << 11) + 1024, 0);
    auto fetch = [&](int t) {
        if (t + lane < t1) next = __ldg(&q.g.taps[t + lane]);
    };
    fetch(q.g.off[k]);
#pragma unroll 1
    for (int t0 = q.g.off[k]; t0 < t1; t0 += 32) {
        const int off = ((next.x >> 11) - 1024) * W + (next.x & 2047) - 1024;
        sm[lane] = make_float2(__int_as_float(inner ? off : next.x), __int_as_float(next.y));
        __syncwarp();
        fetch(t0 + 32);
        const int n = min(32, t1 - t0);
#pragma unroll 1
        for (int h = 0; h < n; h += B) {
            float2 e[B];
            float v[B];
#pragma unroll
            for (int j = 0; j < B; j++) e[j] = sm[h + j];
#pragma unroll
            for (int j = 0; j < B; j++) {
                const int o = __float_as_int(e[j].x);
                v[j] = inner ? __ldg(at + o) : __ldg(plane + tap_site(make_int2(o, 0), y, x, H, W));
            }
#pragma unroll
            for (int j = 0; j < B; j++)
                if (h + j < n) acc = fmaf(e[j].y, v[j], acc);
        }
        __syncwarp();
    }
    return acc;
}

// The warp's marked sites (bit c of a lane's marks: its column c), dealt to the lanes 32
// at a time: `one(y, x, owner, c, valid)` handles a lane's site, for the whole warp, and
// its result goes back to the owner's `take(c, result)`.  slot: the warp's 32 bytes.
template <class One, class Take>
__device__ __forceinline__ void deal_sites(uint8_t* slot, uint32_t marks, int y, int x, One one, Take take)
{
    const int lane = threadIdx.x & 31;
    int before = 0, total = 0;                 // marks of the lanes below, of all
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const uint32_t b = __ballot_sync(0xffffffffu, (marks >> c) & 1);
        before += __popc(b & ((1u << lane) - 1));
        total += __popc(b);
    }
#pragma unroll 1
    for (int base = 0; base < total; base += 32) {
        int r = before - base;
#pragma unroll
        for (int c = 0; c < 4; c++)
            if ((marks >> c) & 1) {
                if (r >= 0 && r < 32) slot[r] = (uint8_t)(4 * lane + c);
                r++;
            }
        __syncwarp();
        const bool valid = base + lane < total;
        const int s = valid ? slot[lane] : 0, owner = s >> 2, c = s & 3;
        const float res = one(__shfl_sync(0xffffffffu, y, owner), __shfl_sync(0xffffffffu, x, owner) + c, owner, c, valid);
        r = before - base;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float v = __shfl_sync(0xffffffffu, res, r & 31);
            if ((marks >> i) & 1) {
                if (r >= 0 && r < 32) take(i, v);
                r++;
            }
        }
        __syncwarp();
    }
}

// (growth bump, alpha test) at one site as the other update kernels compute them from
// the potential u.
__device__ __forceinline__ float2 settled(const SitesParams& q, float u, float m, float sg, float hh)
{
    float gk = 0.f;
    if (sg > 0.f) {
        if (q.fast) {
            const float z = (u - m) * rcp_approx(sg);
            gk = ex2_approx(-0.721347520444481703680f * (z * z));            // -log2(e) / 2
        } else {
            const float z = (u - m) / sg;
            gk = expf(-0.5f * z * z);
        }
    }
    return make_float2(gk, q.e.alpha_on ? u : hh * gk);
}

// (the streaming kernel's minimum of the tests passes NaN over, the others' do not)
__device__ __forceinline__ bool passes(const SitesParams& q, float t)
{
    return q.fast ? !(t <= q.e.eps_u) : t > q.e.eps_u;
}

// How far a test t = h g (or u) at a potential u and |z| may be off: rounding, and the
// potential's du.  With eta = du / s <= 1/64 the bump's ratio at z + d, |d| <= eta, is
// exp(-z d - d^2 / 2): off by at most 2 |z| eta + eta^2 (|z| eta <= 5/4; beyond it both
// bumps are zero).  `wide`: a narrower bump, or a threshold that lies where bumps
// underflow; see test_range.
__device__ __forceinline__ float test_off(const SitesParams& q, float u, float t, float az, float sg, float rs, bool& wide)
{
    // (u below zero by more than rounding: out of the unit interval, and summed directly)
    const float du = fminf(q.g.du, fmaf(q.g.slope, u, q.g.floor));
    wide = false;
    if (q.e.alpha_on) return fmaf(1e-7f, fabsf(u), du);
    const float eta = du * rs;
    wide = sg > 0.f && (eta > 1.f / 64.f || q.tiny_eps);
    return fabsf(t) * fmaf(2e-6f, az * az, fmaf(eta, fmaf(2.f, az, eta), 2e-6f));
}

// The range (low, high) of a `wide` test: a narrow bump's at z -+ eta.
__device__ __forceinline__ float2 test_range(const SitesParams& q, float u, float t, float az, float sg, float hh, float off)
{
    const float eta = fminf(q.g.du, fmaf(q.g.slope, u, q.g.floor)) * rcp_approx(sg);
    if (eta > 1.f / 64.f) {
        const float z0 = fmaxf(az - eta, 0.f), z1 = az + eta;
        const float t0 = hh * ex2_approx(-0.721347520444481703680f * (z0 * z0));
        const float t1 = hh * ex2_approx(-0.721347520444481703680f * (z1 * z1));
        const float r = fabsf(t0) * fmaf(2e-6f, fminf(z0 * z0, 225.f), 2e-6f);
        return make_float2(fminf(t0, t1) - r, fmaxf(t0, t1) + r);
    }
    if (az < 15.f && fabsf(t) < 1e-36f) off = 1e-36f;
    return make_float2(t - off, t + off);
}

// Whether a test may come out either way, and by how much it may be off.
__device__ __forceinline__ bool undecided_test(const SitesParams& q, float u, float t, float az, float sg, float rs, float hh,
                                               float& off)
{
    bool wide;
    off = test_off(q, u, t, az, sg, rs, wide);
    bool open = fabsf(t - q.e.eps_u) < off;    // (an exact test has off = 0)
    if (wide) {
        const float2 r = test_range(q, u, t, az, sg, hh, off);
        open = r.x < q.e.eps_u && q.e.eps_u < r.y;
        off = fmaxf(r.y - t, t - r.x);
    }
    return open;
}

// Kernel k's diffused genes at one site as the kernel divides them that the shape
// otherwise takes (the streaming kernel by the hardware reciprocal).
template <int NP, int RD>
__device__ __forceinline__ void genes_at(const SitesParams& q, const float* P, int k, int y, int x, float* g)
{
    const EpiParams& p = q.e;
    const int H = p.H, W = p.W;
#pragma unroll
    for (int pp = 0; pp < NP; pp++) {
        const float* pl = P + (size_t)(pp * p.kt.K + k) * H * W;
        float s = 0.f, n = 0.f;
#pragma unroll
        for (int dy = -RD; dy <= RD; dy++)
#pragma unroll
            for (int dx = -RD; dx <= RD; dx++) {
                if (dy * dy + dx * dx > RD * RD) continue;
                int yy = y + dy, xx = x + dx;
                yy = yy < 0 ? yy + H : (yy >= H ? yy - H : yy);
                xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
                const float v = __ldg(&pl[(size_t)yy * W + xx]);
                s += v;
                n += v > p.eps_p ? 1.f : 0.f;
            }
        const float r = q.fast ? s * rcp_approx(n) : s / n;
        g[pp] = n > 0.f ? __saturatef(r) : 0.f;
    }
}

// alpha's undecided tests, settled, at the sites of the lanes that want it: kernel
// `first`'s, and the later kernels' where it was not the only one (the whole warp calls it).
template <int LOC, int RD>
__device__ __forceinline__ bool alpha_at(const SitesParams& q, const float* A, const float* P, const float* U, int y, int x,
                                         bool want, int first, bool more, float2* sm)
{
    const EpiParams& p = q.e;
    const int W = p.W, K = p.kt.K;
    const size_t N = (size_t)p.H * W;
    bool ok = want;
    int k = first;                             // (a lane's own; K: done)
#pragma unroll 1
    while (__any_sync(0xffffffffu, ok && k < K)) {
        // the lanes at the warp's lowest kernel go on
        const int kk = __reduce_min_sync(0xffffffffu, ok && k < K ? k : K);
        const bool on = ok && k == kk;
        float g[3] = {0.f, 0.f, 0.f};          // (mu, sigma and, with LOC 7, h)
        if (on) genes_at<LOC == 7 ? 3 : 2, RD>(q, P, kk, y, x, g);
        const float m = g[0], sg = g[1], hh = LOC == 7 ? g[2] : p.kt.h[kk];
        float u = on ? __ldg(&U[(size_t)kk * N + (size_t)y * W + x]) : 0.f;
        float t = settled(q, u, m, sg, hh).y;
        // a lane's first kernel is known to be undecided
        bool open = on;
        if (__any_sync(0xffffffffu, on && kk != first)) {
            const float rs = rcp_approx(sg);
            float off;
            open = on && (kk == first || undecided_test(q, u, t, fabsf((u - m) * rs), sg, rs, hh, off));
        }
        if (q.g.du > 0.f && __any_sync(0xffffffffu, open)) {
            u = direct_sums(q, A, kk, y, x, open, sm);
            if (open) t = settled(q, u, m, sg, hh).y;
        }
        if (on) {
            ok = passes(q, t);
            k = more ? kk + 1 : K;
        }
    }
    return ok;
}

// sum_k of the alpha tests, settled, at the sites of the lanes that want it (a
// Delta_sum(U) decision near its threshold; the whole warp calls it).
template <int LOC, int RD>
__device__ __forceinline__ float tests_at(const SitesParams& q, const float* A, const float* P, const float* U, int y, int x,
                                       bool want, float2* sm)
{
    const EpiParams& p = q.e;
    const int W = p.W, K = p.kt.K;
    const size_t N = (size_t)p.H * W;
    float sum = 0.f;
    for (int k = 0; k < K; k++) {
        float g[3] = {0.f, 0.f, 0.f};
        if (want) genes_at<LOC == 7 ? 3 : 2, RD>(q, P, k, y, x, g);
        const float m = g[0], sg = g[1], hh = LOC == 7 ? g[2] : p.kt.h[k];
        const float u = q.g.du > 0.f ? direct_sums(q, A, k, y, x, want && (sg > 0.f || p.alpha_on), sm)
                                     : (want ? __ldg(&U[(size_t)k * N + (size_t)y * W + x]) : 0.f);
        if (want) sum += settled(q, u, m, sg, hh).y;
    }
    return sum;
}

// LOC: the localized growth genes (LENIA_LOC_* bits).
template <int LOC, int CT, int RD>
__global__ void __launch_bounds__(ES_T, CT > 3 || RD == 2 ? 3 : 4) k_epilogue_sites(const __grid_constant__ SitesParams q)
{
    pdl_enter();
    constexpr int NP = ((LOC & 1) != 0) + ((LOC & 2) != 0) + ((LOC & 4) != 0);
    constexpr int NQ = NP > 0 ? NP : 1;
    constexpr int PMU = (LOC & 1) ? 0 : -1;
    constexpr int PSG = (LOC & 2) ? ((LOC & 1) ? 1 : 0) : -1;
    constexpr int PH = (LOC & 4) ? NP - 1 : -1;
    const EpiParams& p = q.e;
    // statistics: each thread's own sums over its tiles, in compensated pairs (their number
    // grows with the world)
    __shared__ float2 ssum[CT * 5][ES_T];
    __shared__ uint8_t slot[ES_NW][32];
    __shared__ __align__(16) float2 taps[ES_NW][ES_TAPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int H = p.H, W = p.W, K = p.kt.K, C = p.kt.C;
    const size_t N = (size_t)H * W;
    const float eps_p = p.eps_p, eps_u = p.eps_u;
    if (p.partials) {
#pragma unroll
        for (int v = 0; v < CT * 5; v++) ssum[v][threadIdx.x] = make_float2(0.f, 0.f);
    }
    const int per_world = q.tx * q.ty;
    for (int t = blockIdx.x; t < per_world * q.n_worlds; t += gridDim.x) {
        const int wz = t / per_world, tt = t - wz * per_world;
        const int by = tt / q.tx, bx = tt - by * q.tx;
        const float* pA = p.A_list ? p.A_list[wz] : p.A;
        const float* pP = p.P_list ? p.P_list[wz] : p.P;
        float* pAo = p.Aout_list ? p.Aout_list[wz] : p.A_out;
        float* pPo = p.Pout_list ? p.Pout_list[wz] : p.P_out;
        const float* pU = p.U + (size_t)wz * p.u_stride;
        // a warp takes 8 quads of 4 rows and stays together: lanes beyond the world's
        // edge stand on the torus's continuation and store nothing
        const int qx = lane & (ES_Q - 1), ry = lane / ES_Q;
        const int xq = (bx * ES_Q + qx) * 4, yq = by * ES_Y + warp * (32 / ES_Q) + ry;
        const bool in = xq < W && yq < H;
        const int x = in || xq < W ? xq : xq % W, y = yq < H ? yq : yq % H;
        {
            const int i0 = y * W + x;
            auto quad = [&](const float* base) { return __ldg(reinterpret_cast<const float4*>(base)); };
            // Radius 1: the quads around a quad are other lanes' own (shuffles), but for
            // the warp's rim, whose lanes also load the row above or below and
            // the column beside.  Radius 2 loads its neighbours itself (row
            // offsets from row y, columns left and right).
            const bool rim_y = ry == 0 || ry == 32 / ES_Q - 1, rim_x = qx == 0 || qx == ES_Q - 1;
            int ro[2 * RD + 1], xl[2], xr[2], ie = i0, is = i0;
            if constexpr (RD == 1) {
                const int yn = ry == 0 ? (y == 0 ? H - 1 : y - 1) : (y == H - 1 ? 0 : y + 1);
                ie = yn * W + x;
                is = y * W + (qx == 0 ? (x == 0 ? W - 1 : x - 1) : (x + 4 == W ? 0 : x + 4));
            }
            if constexpr (RD == 2) {
#pragma unroll
                for (int j = 0; j <= 2 * RD; j++) {
                    const int r = y + j - RD;
                    ro[j] = (j - RD + (r < 0 ? H : (r >= H ? -H : 0))) * W;
                }
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    xl[i] = -1 - i + (x - 1 - i < 0 ? W : 0);
                    xr[i] = 4 + i - (x + 4 + i >= W ? W : 0);
                }
            }
            // a kernel's planes and potential are fetched one kernel ahead
            struct Pre {
                float4 c, e;
                float s;
            } nx[NQ];
            float4 nu = make_float4(0.f, 0.f, 0.f, 0.f);
            auto fetch = [&](const float* plane, Pre& o) {
                o.c = quad(plane + i0);
                if constexpr (RD == 1) {
                    if (rim_y) o.e = quad(plane + ie);
                    if (rim_x) o.s = __ldg(plane + is);
                }
            };
            auto gather = [&](const Pre& o, const float* plane, Stencil<RD>& s) {
                if constexpr (RD == 1) {
                    const float c[4] = {o.c.x, o.c.y, o.c.z, o.c.w}, e[4] = {o.e.x, o.e.y, o.e.z, o.e.w};
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const float u = __shfl_up_sync(0xffffffffu, c[i], ES_Q), d = __shfl_down_sync(0xffffffffu, c[i], ES_Q);
                        s.v[0][1 + i] = ry == 0 ? e[i] : u;
                        s.v[1][1 + i] = c[i];
                        s.v[2][1 + i] = ry == 32 / ES_Q - 1 ? e[i] : d;
                    }
                    const float l = __shfl_up_sync(0xffffffffu, c[3], 1), r = __shfl_down_sync(0xffffffffu, c[0], 1);
                    s.v[1][0] = qx == 0 ? o.s : l;
                    s.v[1][5] = qx == ES_Q - 1 ? o.s : r;
                } else {
                    s.load(plane + i0, ro, xl, xr, o.c);
                }
            };
            bool live = in;
            if constexpr (NP > 0) {
                fetch(pP, nx[0]);
                if (q.gate) {
                    if constexpr (RD == 1) {
                        float m = fmaxf(fmaxf(nx[0].c.x, nx[0].c.y), fmaxf(nx[0].c.z, nx[0].c.w));
                        if (rim_y) m = fmaxf(m, fmaxf(fmaxf(nx[0].e.x, nx[0].e.y), fmaxf(nx[0].e.z, nx[0].e.w)));
                        if (rim_x) m = fmaxf(m, nx[0].s);
                        live = m > eps_p;                   // (of the warp, below)
                    } else {
                        Stencil<RD> s;
                        gather(nx[0], pP, s);
                        live = s.any_above(eps_p);
                    }
                }
            }
            float acc[CT][4];
#pragma unroll
            for (int c = 0; c < CT; c++)
#pragma unroll
                for (int i = 0; i < 4; i++) acc[c][i] = 0.f;
            bool al[4] = {in, in, in, in};
            float tsum[4] = {0.f, 0.f, 0.f, 0.f}, tband[4] = {0.f, 0.f, 0.f, 0.f};
            bool wrote = false;                     // a non-zero gene went out already
            uint32_t undecided = 0, many = 0, first = 0;    // sites with tests to be settled; with several; their first kernels
            int k = 0;
            const bool warp_live = __any_sync(0xffffffffu, live);
            if (NP > 0 && !warp_live) al[0] = al[1] = al[2] = al[3] = false;
            if (warp_live) {
                const size_t KN = (size_t)K * N;
                const float* up = pU + i0;
                const float* gp = pP;               // kernel k's first plane
                float* go = pPo + i0;
                bool want = in;                     // something left to compute for this quad
                nu = quad(up);
#pragma unroll
                for (int pp = 1; pp < NP; pp++) fetch(gp + pp * KN, nx[pp]);
#pragma unroll 1
                for (; k < K; k++) {
                    float ph[NQ][4], u[4], gk[4], tk[4];
                    const float km = p.kt.mu[k], ks = p.kt.sigma[k], kh = p.kt.h[k];
                    auto mu_of = [&](int c) { return PMU >= 0 ? ph[PMU >= 0 ? PMU : 0][c] : km; };
                    auto sg_of = [&](int c) { return PSG >= 0 ? ph[PSG >= 0 ? PSG : 0][c] : ks; };
                    auto h_of = [&](int c) { return PH >= 0 ? ph[PH >= 0 ? PH : 0][c] : kh; };
                    uint32_t now = 0;               // undecided tests: they pass for now
                    Pre cur[NQ];
#pragma unroll
                    for (int pp = 0; pp < NP; pp++) cur[pp] = nx[pp];
                    u[0] = nu.x, u[1] = nu.y, u[2] = nu.z, u[3] = nu.w;
                    up += N;
                    if (k + 1 < K) {
                        nu = quad(up);
#pragma unroll
                        for (int pp = 0; pp < NP; pp++) fetch(gp + pp * KN + N, nx[pp]);
                    }
#pragma unroll
                    for (int pp = 0; pp < NP; pp++) {
                        Stencil<RD> s;
                        gather(cur[pp], gp + pp * KN, s);
                        s.diffused(eps_p, ph[pp]);
#pragma unroll
                        for (int c = 0; c < 4; c++) al[c] = al[c] & (ph[pp][c] > eps_p);
                    }
                    if (want) {
#pragma unroll
                        for (int c = 0; c < 4; c++) {
                            const float sg = sg_of(c);
                            const float rs = rcp_approx(sg), z = (u[c] - mu_of(c)) * rs, z2 = z * z;
                            const float e = ex2_approx(-0.721347520444481703680f * z2);      // -log2(e) / 2
                            gk[c] = sg > 0.f ? e : 0.f;
                            tk[c] = p.alpha_on ? u[c] : h_of(c) * gk[c];
                            if (NP > 0) {
                                float off;
                                const bool open = undecided_test(q, u[c], tk[c], fabsf(z), sg, rs, h_of(c), off);
                                if (p.empty_out) tband[c] += sg > 0.f || p.alpha_on ? off : 0.f;
                                now |= (open ? 1u : 0u) << c;
                            }
                        }
                        if (NP > 0 && now) {
                            many |= undecided & now;
#pragma unroll
                            for (int c = 0; c < 4; c++)
                                if ((now & ~undecided) >> c & 1) first |= (uint32_t)k << (8 * c);
                            undecided |= now;
                        }
                    }
                    float G[4];
                    if (want) {
#pragma unroll
                        for (int c = 0; c < 4; c++) {
                            if (NP > 0) al[c] = al[c] & (passes(q, tk[c]) | ((now >> c) & 1));
                            tsum[c] += tk[c];
                            G[c] = p.growth_form == 0 ? fmaf(2.f * gk[c], h_of(c), -h_of(c)) : h_of(c) * gk[c];
                        }
                        const int d = p.kt.dst[k];
#pragma unroll
                        for (int cc = 0; cc < CT; cc++)
                            if (CT == 1 || cc == d)
#pragma unroll
                                for (int c = 0; c < 4; c++) acc[cc][c] += G[c];
                    }
                    if (NP > 0) {
                        const bool any = al[0] | al[1] | al[2] | al[3];
                        wrote |= any;
                        if (in)
#pragma unroll
                        for (int pp = 0; pp < NP; pp++)
                            *reinterpret_cast<float4*>(go + pp * KN) =
                                make_float4(al[0] ? ph[pp][0] : 0.f, al[1] ? ph[pp][1] : 0.f,
                                            al[2] ? ph[pp][2] : 0.f, al[3] ? ph[pp][3] : 0.f);
                        gp += N;
                        go += N;
                        // alpha is false at all four sites: nothing more to compute, unless
                        // Delta_sum wants every kernel's growth
                        want = want && (any || p.empty_out);
                        if (!__any_sync(0xffffffffu, want)) {
                            k++;
                            break;
                        }
                    }
                }
            }
            if (NP > 0) {
                // sites that hang on undecided tests
                const uint32_t open = undecided & (al[0] | (al[1] << 1) | (al[2] << 2) | (al[3] << 3));
                if (__any_sync(0xffffffffu, open != 0)) {
                    uint32_t lost = 0;
                    deal_sites(
                        slot[warp], open, y, x,
                        [&](int ys, int xs, int owner, int c, bool valid) {
                            const int k0 = (__shfl_sync(0xffffffffu, first, owner) >> (8 * c)) & 255;
                            const bool more = (__shfl_sync(0xffffffffu, many, owner) >> c) & 1;
                            return alpha_at<LOC, RD>(q, pA, pP, pU, ys, xs, valid, k0, more, taps[warp]) ? 1.f : 0.f;
                        },
                        [&](int c, float ok) { lost |= (ok == 0.f ? 1u : 0u) << c; });
#pragma unroll
                    for (int c = 0; c < 4; c++) al[c] = al[c] & !((lost >> c) & 1);
                }
            }
            if (NP > 0 && in) {
                const bool all = al[0] & al[1] & al[2] & al[3], any = al[0] | al[1] | al[2] | al[3];
                const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int pp = 0; pp < NP; pp++) {
                    float* o = pPo + (size_t)pp * K * N + i0;
                    // planes of the kernels that were not reached (alpha is false)
                    for (int j = k; j < K; j++) *reinterpret_cast<float4*>(o + (size_t)j * N) = z4;
                    // planes written before alpha was known to be false
                    if (wrote && !any)
                        for (int j = 0; j < k; j++) *reinterpret_cast<float4*>(o + (size_t)j * N) = z4;
                    else if (wrote && !all)
                        for (int j = 0; j < k; j++)
#pragma unroll
                            for (int c = 0; c < 4; c++)
                                if (!al[c]) o[(size_t)j * N + c] = 0.f;
                }
            }
#pragma unroll
            for (int c = 0; c < CT; c++) {
                if (c >= C || !in) break;
                const float4 a4 = __ldg(reinterpret_cast<const float4*>(pA + (size_t)c * N + i0));
                const float a[4] = {a4.x, a4.y, a4.z, a4.w};
                float o[4];
#pragma unroll
                for (int i = 0; i < 4; i++) o[i] = __saturatef(a[i] + p.dt * ((NP == 0 || al[i]) ? acc[c][i] : p.acc0[c]));
                *reinterpret_cast<float4*>(pAo + (size_t)c * N + i0) = make_float4(o[0], o[1], o[2], o[3]);
                if (p.partials) {
                    // (the tables start at any float: scalar loads)
                    const float* sx = p.sin_x + x;
                    const float* cx = p.cos_x + x;
                    const float m = (o[0] + o[1]) + (o[2] + o[3]);
                    float2* a5 = &ssum[c * 5][threadIdx.x];
                    auto add = [&](int v, float t) {       // (two-sum, the errors collected in .y)
                        const float2 a = a5[v * ES_T];
                        const float h = a.x + t, b = h - a.x;
                        a5[v * ES_T] = make_float2(h, a.y + ((a.x - (h - b)) + (t - b)));
                    };
                    add(0, m);
                    add(1, m * __ldg(&p.sin_y[y]));
                    add(2, m * __ldg(&p.cos_y[y]));
                    add(3, (o[0] * __ldg(sx) + o[1] * __ldg(sx + 1)) + (o[2] * __ldg(sx + 2) + o[3] * __ldg(sx + 3)));
                    add(4, (o[0] * __ldg(cx) + o[1] * __ldg(cx + 1)) + (o[2] * __ldg(cx + 2) + o[3] * __ldg(cx + 3)));
                }
            }
            if (in && p.alpha_out)
                *reinterpret_cast<uchar4*>(p.alpha_out + i0) =
                    NP == 0 ? make_uchar4(1, 1, 1, 1) : make_uchar4(al[0], al[1], al[2], al[3]);
            // (no band: every test is exactly the direct route's, and so is their sum)
            if (NP > 0 && p.empty_out) {
                uint32_t close = 0;
#pragma unroll
                for (int c = 0; c < 4; c++)
                    close |= (in && tband[c] > 0.f && fabsf(tsum[c] - eps_u) <= tband[c] + 1e-6f ? 1u : 0u) << c;
                if (__any_sync(0xffffffffu, close != 0))
                    deal_sites(
                        slot[warp], close, y, x,
                        [&](int ys, int xs, int, int, bool valid) { return tests_at<LOC, RD>(q, pA, pP, pU, ys, xs, valid, taps[warp]); },
                        [&](int c, float t) {
#pragma unroll
                            for (int i = 0; i < 4; i++)
                                if (c == i) tsum[i] = t;
                        });
            }
            if (in && p.empty_out)
                *reinterpret_cast<uchar4*>(p.empty_out + i0) =
                    make_uchar4(!(tsum[0] > eps_u), !(tsum[1] > eps_u), !(tsum[2] > eps_u), !(tsum[3] > eps_u));
        }
    }
    if (p.partials) {
        // one warp per value: lanes, then a shuffle tree, in compensated pairs
        __syncthreads();
        for (int v = warp; v < C * 5; v += ES_NW) {
            float2 s = make_float2(0.f, 0.f);
            for (int i = lane; i < ES_T; i += 32) s = ff_add(s, ssum[v][i]);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) s = ff_add(s, ff_shfl_down(s, off));
            if (lane == 0) p.partials[(size_t)blockIdx.x * C * 5 + v] = s;
        }
    }
}

template <int LOC, int CT, int RD>
cudaError_t launch_sites(SitesParams& q, int max_blocks, cudaStream_t s, int* n_blocks)
{
    const long long tiles = (long long)q.tx * q.ty * q.n_worlds;
    const int blocks = (int)(tiles < max_blocks ? tiles : max_blocks);
    if (n_blocks) *n_blocks = blocks;
    launch_pdl(k_epilogue_sites<LOC, CT, RD>, dim3(blocks), dim3(ES_T), 0, s, q);
    return cudaGetLastError();
}

template <int LOC, int RD>
cudaError_t launch_sites_c(SitesParams& q, int max_blocks, cudaStream_t s, int* n_blocks)
{
    const int C = q.e.kt.C;
    if (C == 1) return launch_sites<LOC, 1, RD>(q, max_blocks, s, n_blocks);
    if (C <= 3) return launch_sites<LOC, 3, RD>(q, max_blocks, s, n_blocks);
    return launch_sites<LOC, kMaxChannels, RD>(q, max_blocks, s, n_blocks);
}

}  // namespace

bool epilogue_sites_supported(const EpiParams& p)
{
    if (p.n_rings || p.p_kern >= 0 || (size_t)p.H * p.W >= (1u << 30)) return false;
    const int loc = (p.p_mu >= 0 ? 1 : 0) | (p.p_sigma >= 0 ? 2 : 0) | (p.p_h >= 0 ? 4 : 0);
    return (loc == 0 && !p.empty_out) || ((loc == 3 || loc == 7) && p.maintain && p.eps_p == 0.f && (p.r_diff == 1 || p.r_diff == 2));
}

bool epilogue_gated(const EpiParams& p)
{
    return p.maintain && p.n_p > 0 && p.eps_p >= 0.f && !p.empty_out;
}

cudaError_t launch_epilogue_sites(const EpiParams& p, bool fast, const GuardParams* guard, int n_worlds, int max_blocks,
                                  cudaStream_t s, int* n_blocks)
{
    if (!epilogue_sites_supported(p) || n_worlds < 1 || max_blocks < 1) return cudaErrorInvalidValue;
    SitesParams q;
    memset(&q, 0, sizeof(q));
    q.e = p;
    if (guard) q.g = *guard;
    q.n_worlds = n_worlds;
    q.tx = (p.W + 4 * ES_Q - 1) / (4 * ES_Q);
    q.ty = (p.H + ES_Y - 1) / ES_Y;
    q.gate = epilogue_gated(p);
    q.tiny_eps = fabsf(p.eps_u) < 1e-30f;
    q.fast = fast;
    if (p.n_p == 0) return launch_sites_c<0, 0>(q, max_blocks, s, n_blocks);
    if (p.r_diff == 1)
        return p.n_p == 2 ? launch_sites_c<3, 1>(q, max_blocks, s, n_blocks) : launch_sites_c<7, 1>(q, max_blocks, s, n_blocks);
    return p.n_p == 2 ? launch_sites_c<3, 2>(q, max_blocks, s, n_blocks) : launch_sites_c<7, 2>(q, max_blocks, s, n_blocks);
}

}  // namespace lenia

// Spectral convolution in overlapping tiles (convolution theorem, note after
// Algorithm 2 of arXiv 2304.05639), one launch for every kernel of a world.
//
// A block takes an N x N window of one channel (N = 64 or 128) that starts R
// sites before its output tile and wraps around the torus, transforms it
// once in shared memory, and for each kernel reading that channel multiplies
// by the kernel's spectrum (real: the kernels are point symmetric) and
// transforms back.  The window's circular convolution equals the torus's on
// the (N - 2R) x (N - 2R) sites whose neighbourhood lies inside the window
// (overlap-save), and those are written.  Where a side of the world is N itself
// the window is the whole torus along that axis and nothing overlaps.
//
// The window's rows are real and travel as N/2 complex values; element 0 of a
// row spectrum packs the two real values X[0] and X[N/2] as (re, im).  Both 2-D
// transforms are four in-place passes over the [N][N/2] buffer, each pass one
// radix-16, -8 or -4 butterfly per task with a barrier after it:
//   forward  rows: 8 over m2, RR over m1 + even/odd split;  columns: 8, CA
//   inverse  columns: product + CA, 8;  rows: recombination + RR, 8
// with N = 8 CA and N/2 = 8 RR.  In place means that a pass writes the
// elements it read, so indices leave in digit-swapped order: row y = n1 + CA q
// holds sub-transform q of residue n1 in the middle of a column transform and
// image row y at its end; column position m1 8 + j holds the middle of a row
// transform, column kx its end.
//
// A warp's tasks differ only in the lane's column (column passes) or row (row
// passes), so the twiddles of a task are the same for all lanes: compile-time
// constants in the row passes, broadcast shared loads in the column passes.
// The forward spectrum stays in tensor memory (TMEM), each thread's share in
// its own lane, so that one 64 KB buffer serves all transforms and three
// blocks fit on an SM.
//
// What bounds it: the FP32 pipes and instruction issue (about 1500 FP32
// operations per thread and inverse transform, against 7 shared-memory passes).
// 1080 x 1920, 15 kernels R = 13: 97 us, 52 to 66 where the gate skips half of the
// windows (direct sums 1135); 2048^2, 15 kernels R = 5, gated: 107 us (102 without
// the look at its values; direct sums 415); 256^2, 15 kernels: 11 us (three FFT
// passes 14).
#include <math.h>

#include <utility>

#include "fft_core.cuh"
#include "lenia_internal.cuh"
#include "ptx_util.cuh"

namespace lenia {
namespace {

// cos(2 pi m / n) and sin(2 pi m / n) at compile time: octant reduction on the
// integers (n a multiple of 8), then the Taylor series on [0, pi/4].
constexpr double kTau = 6.283185307179586476925286766559;
__host__ __device__ constexpr double ct_series(double x, int first)        // first = 0: cos, 1: sin
{
    double t = first ? x : 1.0, s = t;
    for (int i = first + 1; i < first + 24; i += 2) {
        t *= -x * x / ((double)i * (i + 1));
        s += t;
    }
    return s;
}
__host__ __device__ constexpr double ct_cos(int m, int n)
{
    m %= n;
    if (m < 0) m += n;
    if (2 * m > n) m = n - m;
    if (4 * m > n) return -ct_cos(n / 2 - m, n);
    if (8 * m > n) return ct_series(kTau * (n / 4 - m) / n, 1);
    return ct_series(kTau * m / n, 0);
}
__host__ __device__ constexpr double ct_sin(int m, int n) { return ct_cos(m - n / 4, n); }

template <class F, int... I>
__device__ __forceinline__ void for_seq(F f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F f)
{
    for_seq(f, std::make_integer_sequence<int, N>{});
}

// a exp(2 pi i Q / NN) with compile-time Q
template <int Q, int NN>
__device__ __forceinline__ float2 ctw(float2 a)
{
    constexpr int q = ((Q % NN) + NN) % NN;
    if constexpr (q == 0) return a;
    else if constexpr (4 * q == NN) return make_float2(-a.y, a.x);
    else if constexpr (2 * q == NN) return make_float2(-a.x, -a.y);
    else if constexpr (4 * q == 3 * NN) return make_float2(a.y, -a.x);
    else {
        constexpr float c = (float)ct_cos(q, NN), s = (float)ct_sin(q, NN);
        return make_float2(a.x * c - a.y * s, a.x * s + a.y * c);
    }
}

template <int N, int NT = 2 * N>
struct TC {
    static constexpr int M = N / 2;            // complex values per row
    static constexpr int CA = N / 8;           // column transform: CA x 8
    static constexpr int RR = M / 8;           // row transform: RR x 8
    static constexpr int T = NT;               // threads: 2 N or 4 N (see launch_n)
    static constexpr int NW = T / 32;          // warps
    static constexpr int CH = M / 32;          // 32-column halves
    static constexpr int TMEM = N == 128 ? 128 : 32;      // TMEM columns of a block
    static constexpr int PITCH = M * 8;        // bytes per row
    static constexpr size_t SMEM = (size_t)N * M * 8 + 3 * (size_t)N * 8;
};

// Byte offset of (row, col) in the buffer: the column index is XORed with its
// own bits 3.. and with the reversed low four row bits, which spreads both
// 16 consecutive rows of one column (row passes) and 8 columns 8 apart in
// two adjacent rows (first forward and last inverse pass) over all banks.
__device__ __forceinline__ int row_sw(int y)
{
    return ((y & 1) << 3) | ((y & 2) << 1) | ((y & 4) >> 1) | ((y & 8) >> 3);
}
__device__ __forceinline__ int col_sw(int c) { return c ^ ((c >> 3) & 7); }
template <int N>
__device__ __forceinline__ int at(int row, int col)
{
    return row * TC<N>::PITCH + (col_sw(col) ^ row_sw(row)) * 8;
}
__device__ __forceinline__ float2 ld2(const unsigned char* b, int off) { return *reinterpret_cast<const float2*>(b + off); }
__device__ __forceinline__ void st2(unsigned char* b, int off, float2 v) { *reinterpret_cast<float2*>(b + off) = v; }

// Row pass of task t (positions j = t and its mirror) of row y, forward:
// twiddle, radix RR over m1, and the even/odd split of the real rows
//   X[q] = s + d, X[M - q] = conj(s - d),
//   s = Z[q] + conj Z[M-q], d = -i w^q (Z[q] - conj Z[M-q]), w = exp(-2 pi i / N)
// (twice the spectrum; the kernel spectra carry the factor 1/2).
template <int N, int t>
__device__ __forceinline__ void rows_fwd(unsigned char* buf, int y)
{
    constexpr int RR = TC<N>::RR, M = TC<N>::M;
    constexpr int jA = t, jB = t == 0 ? 4 : 8 - t;
    const int base = y * TC<N>::PITCH + row_sw(y) * 8;
    float2 a[RR], b[RR];
    static_for<RR>([&](auto I) {
        constexpr int m1 = decltype(I)::value;
        constexpr int cA = m1 * 8 + (jA ^ (m1 & 7)), cB = m1 * 8 + (jB ^ (m1 & 7));
        a[m1] = ctw<-m1 * jA, M>(ld2(buf, base ^ (cA * 8)));
        b[m1] = ctw<-m1 * jB, M>(ld2(buf, base ^ (cB * 8)));
    });
    DFT<RR, false, true>::run(a);
    DFT<RR, false, true>::run(b);
    auto split = [&](auto Q, float2& zk, float2& zm) {
        const float2 s = make_float2(zk.x + zm.x, zk.y - zm.y);
        const float2 e = make_float2(zk.x - zm.x, zk.y + zm.y);
        const float2 d = ctw<-decltype(Q)::value - N / 4, N>(e);          // -i w^q e
        zk = make_float2(s.x + d.x, s.y + d.y);
        zm = make_float2(s.x - d.x, -(s.y - d.y));
    };
    if constexpr (t == 0) {
        a[0] = make_float2(2.f * (a[0].x + a[0].y), 2.f * (a[0].x - a[0].y));
        // q = M / 2 is its own mirror: X = 2 conj Z
        a[RR / 2] = make_float2(2.f * a[RR / 2].x, -2.f * a[RR / 2].y);
        static_for<RR / 2 - 1>([&](auto I) {
            constexpr int r = decltype(I)::value + 1;
            split(std::integral_constant<int, 8 * r>{}, a[r], a[RR - r]);
        });
        static_for<RR / 2>([&](auto I) {
            constexpr int r = decltype(I)::value;
            split(std::integral_constant<int, 4 + 8 * r>{}, b[r], b[RR - 1 - r]);
        });
    } else {
        static_for<RR>([&](auto I) {
            constexpr int r = decltype(I)::value;
            split(std::integral_constant<int, jA + 8 * r>{}, a[r], b[RR - 1 - r]);
        });
    }
    static_for<RR>([&](auto I) {
        constexpr int r = decltype(I)::value;
        constexpr int cA = r * 8 + (jA ^ (r & 7)), cB = r * 8 + (jB ^ (r & 7));
        st2(buf, base ^ (cA * 8), a[r]);
        st2(buf, base ^ (cB * 8), b[r]);
    });
}

// The same task of the inverse transform: recombination
//   Z[q] = s + i d, Z[M - q] = conj(s - i d),
//   s = X[q] + conj X[M-q], d = conj(w^q) (X[q] - conj X[M-q]),
// radix RR over r, twiddle.
template <int N, int t>
__device__ __forceinline__ void rows_inv(unsigned char* buf, int y)
{
    constexpr int RR = TC<N>::RR, M = TC<N>::M;
    constexpr int jA = t, jB = t == 0 ? 4 : 8 - t;
    const int base = y * TC<N>::PITCH + row_sw(y) * 8;
    float2 a[RR], b[RR];
    static_for<RR>([&](auto I) {
        constexpr int r = decltype(I)::value;
        constexpr int cA = r * 8 + (jA ^ (r & 7)), cB = r * 8 + (jB ^ (r & 7));
        a[r] = ld2(buf, base ^ (cA * 8));
        b[r] = ld2(buf, base ^ (cB * 8));
    });
    auto join = [&](auto Q, float2& xk, float2& xm) {
        const float2 s = make_float2(xk.x + xm.x, xk.y - xm.y);
        const float2 e = make_float2(xk.x - xm.x, xk.y + xm.y);
        const float2 d = ctw<decltype(Q)::value + N / 4, N>(e);           // i conj(w^q) e
        xk = make_float2(s.x + d.x, s.y + d.y);
        xm = make_float2(s.x - d.x, -(s.y - d.y));
    };
    if constexpr (t == 0) {
        a[0] = make_float2(a[0].x + a[0].y, a[0].x - a[0].y);
        a[RR / 2] = make_float2(2.f * a[RR / 2].x, -2.f * a[RR / 2].y);
        static_for<RR / 2 - 1>([&](auto I) {
            constexpr int r = decltype(I)::value + 1;
            join(std::integral_constant<int, 8 * r>{}, a[r], a[RR - r]);
        });
        static_for<RR / 2>([&](auto I) {
            constexpr int r = decltype(I)::value;
            join(std::integral_constant<int, 4 + 8 * r>{}, b[r], b[RR - 1 - r]);
        });
    } else {
        static_for<RR>([&](auto I) {
            constexpr int r = decltype(I)::value;
            join(std::integral_constant<int, jA + 8 * r>{}, a[r], b[RR - 1 - r]);
        });
    }
    DFT<RR, true, true>::run(a);
    DFT<RR, true, true>::run(b);
    static_for<RR>([&](auto I) {
        constexpr int m1 = decltype(I)::value;
        constexpr int cA = m1 * 8 + (jA ^ (m1 & 7)), cB = m1 * 8 + (jB ^ (m1 & 7));
        st2(buf, base ^ (cA * 8), ctw<m1 * jA, M>(a[m1]));
        st2(buf, base ^ (cB * 8), ctw<m1 * jB, M>(b[m1]));
    });
}

// Radix-8 column pass (no twiddle) over the rows n1 + CA q of column c.
template <int N, bool INV>
__device__ __forceinline__ void cols8(unsigned char* buf, int n1, int c)
{
    constexpr int CA = TC<N>::CA;
    float2 v[8];
    // the swizzle takes the low four row bits: n1, or n1 + 8 (q & 1) where CA = 8
    const int o0 = at<N>(n1, c), o1 = at<N>(n1 + CA, c) - CA * TC<N>::PITCH;
#pragma unroll
    for (int q = 0; q < 8; q++) v[q] = ld2(buf, ((q & 1) ? o1 : o0) + q * CA * TC<N>::PITCH);
    DFT<8, INV, true>::run(v);
#pragma unroll
    for (int q = 0; q < 8; q++) st2(buf, ((q & 1) ? o1 : o0) + q * CA * TC<N>::PITCH, v[q]);
}

// The largest magnitude of three, NaN if one is NaN.
__device__ __forceinline__ float max_abs(float a, float b, float c)
{
    float d;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__device__ __forceinline__ int wrap_any(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

struct Window {                     // the tile of a block
    TileGeom g;
    int x0, y0;                     // first output site
    int c, lane, warp;
};

// Forward transform of one plane's window up to the last column pass; stops and
// returns true if the window holds a value beyond the limit.
template <int N, int NT>
__device__ __forceinline__ bool forward_start(const TileParams& p, const float* plane, const Window& w,
                                              unsigned char* buf)
{
    using X = TC<N, NT>;
    const int lane = w.lane, warp = w.warp;
    const bool inside = w.x0 >= w.g.halo_x && w.x0 - w.g.halo_x + N <= p.W && w.y0 >= w.g.halo_y &&
                        w.y0 - w.g.halo_y + N <= p.H;
    const int m1 = lane % X::RR;
    float largest = 0.f;
    {
        // rows: radix 8 over m2 of the pairs m1 + RR m2, straight from global
        // memory; window index i stands for site x0 + i, or x0 + i - N beyond the cut
        int gx[8];
#pragma unroll
        for (int m2 = 0; m2 < 8; m2++) {
            const int i = 2 * (m1 + X::RR * m2);
            gx[m2] = w.x0 + (i < w.g.cut_x ? i : i - N);
            if (!inside) gx[m2] = wrap_any(gx[m2], p.W);
        }
        constexpr int RPW = 32 / X::RR;                   // rows per warp
#pragma unroll 1
        for (int i = 0; i < N / (RPW * X::NW); i++) {
            const int y = (warp + i * X::NW) * RPW + lane / X::RR;
            int gy = w.y0 + (y < w.g.cut_y ? y : y - N);
            if (!inside) gy = wrap_any(gy, p.H);
            const float* row = plane + (size_t)gy * p.W;
            float2 v[8];
            if (p.vec2) {
#pragma unroll
                for (int m2 = 0; m2 < 8; m2++) v[m2] = __ldg(reinterpret_cast<const float2*>(row + gx[m2]));
            } else {
#pragma unroll
                for (int m2 = 0; m2 < 8; m2++) v[m2] = make_float2(__ldg(row + gx[m2]), __ldg(row + gx[m2] + 1));
            }
#pragma unroll
            for (int m2 = 0; m2 < 8; m2++)
                largest = max_abs(largest, v[m2].x - p.centre, v[m2].y - p.centre);
            DFT<8, false, true>::run(v);
            const int base = y * X::PITCH + ((m1 * 8 + (m1 & 7)) ^ row_sw(y)) * 8;
#pragma unroll
            for (int j = 0; j < 8; j++) st2(buf, base ^ (j * 8), v[j]);
        }
    }
    if (__syncthreads_or(p.dw && !(largest <= p.reach))) return true;
    // rows: radix RR over m1 and the real split; warp-uniform t
#pragma unroll 1
    for (int u = warp; u < 4 * (N / 32); u += X::NW) {
        const int y = (u >> 2) * 32 + lane;
        switch (u & 3) {
            case 0: rows_fwd<N, 0>(buf, y); break;
            case 1: rows_fwd<N, 1>(buf, y); break;
            case 2: rows_fwd<N, 2>(buf, y); break;
            default: rows_fwd<N, 3>(buf, y); break;
        }
    }
    __syncthreads();
    // columns: radix 8 over q (rows n1 + CA q)
#pragma unroll 1
    for (int u = warp; u < X::CA * X::CH; u += X::NW) cols8<N, false>(buf, u % X::CA, (u / X::CA) * 32 + lane);
    __syncthreads();
    return false;
}

// Kernel k's direct sum over the plane at (y, x), in k_direct_conv's order.
__device__ __forceinline__ float window_sum(const TileParams& p, const float* plane, int k, int y, int x)
{
    const int R = p.dR[k];
    const float* w = p.dw + p.dw_off[k];       // [dx + R][dy + R]
    const int* yr = p.yr + p.yr_off[k];
    float acc = 0.f;
#pragma unroll 1
    for (int dx = -R; dx <= R; dx++) {
        const int r = __ldg(&yr[dx + R]);
        const float* wc = w + (dx + R) * (2 * R + 1) + R;
        const float* col = plane + wrap_any(x + dx, p.W);
#pragma unroll 1
        for (int dy = -r; dy <= r; dy++) acc = fmaf(__ldg(&wc[dy]), __ldg(col + (size_t)wrap_any(y + dy, p.H) * p.W), acc);
    }
    return acc;
}

// The output tile by direct sums, for a window that holds a value beyond the limit.
// (Inline: as a call it cost the 64^2 windows' passes spills, 2048^2 with R = 5
// 340 against 330 us a step.)
// Kernels t0 .. t1 - 1 of channel c; ADJ: their sum added to the channel's plane.
template <bool ADJ>
__device__ __forceinline__ void window_direct(const TileParams& p, int c, int t0, int t1, int x0, int y0, int rows, int xend)
{
    const size_t HW = (size_t)p.H * p.W;
#pragma unroll 1
    for (int i = threadIdx.x; i < rows * xend; i += blockDim.x) {
        const int y = y0 + i / xend, x = x0 + i % xend;
        const size_t o = (size_t)y * p.W + x;
        float sum = 0.f;
        for (int t = t0; t < t1; t++) {
            const int k = p.per_plane ? c : p.klist[c][t];
            const float u = window_sum(p, p.A + (ADJ ? k : c) * HW, k, y, x);
            if (ADJ) sum += u;
            else p.U[k * HW + o] = u;
        }
        if (ADJ) p.U[c * HW + o] = p.add ? __ldg(p.add + c * HW + o) + sum : sum;
    }
}

// Last forward column pass of (column c, residue b): twiddle w_N^(n1 b), radix CA over
// n1; v[a] is the spectrum at row a 8 + b.
template <int N>
__device__ __forceinline__ void cols_fwd(const unsigned char* buf, const float2* twc, int c, int b, float2* v)
{
    using X = TC<N>;
#pragma unroll
    for (int n1 = 0; n1 < X::CA; n1++) {
        v[n1] = ld2(buf, at<N>(n1 + X::CA * b, c));
        if (n1) v[n1] = cmul(v[n1], twc[b * X::CA + n1]);
    }
    DFT<X::CA, false, true>::run(v);
}

// First inverse column pass, the reverse of cols_fwd (it writes the elements that one read).
template <int N>
__device__ __forceinline__ void cols_inv(unsigned char* buf, const float2* twc, int c, int b, float2* v)
{
    using X = TC<N>;
    DFT<X::CA, true, true>::run(v);
#pragma unroll
    for (int n1 = 0; n1 < X::CA; n1++)
        st2(buf, at<N>(n1 + X::CA * b, c), n1 ? cmulc(v[n1], twc[b * X::CA + n1]) : v[n1]);
}

// Forward transform; task i's CA spectrum values go to `sink(i, c, b, v)`.  Returns
// false, without having called it, if the window holds a value beyond the limit.
template <int N, int NT, int UNR, class Sink>
__device__ __forceinline__ bool forward(const TileParams& p, const float* plane, const Window& w, unsigned char* buf,
                                        const float2* twc, Sink sink)
{
    using X = TC<N, NT>;
    if (forward_start<N, NT>(p, plane, w, buf)) return false;
    constexpr int TASKS = 8 * X::CH / X::NW;             // per warp
#pragma unroll UNR
    for (int i = 0; i < TASKS; i++) {
        const int u = w.warp + i * X::NW;
        const int b = u % 8, c = (u / 8) * 32 + w.lane;
        float2 v[X::CA];
        cols_fwd<N>(buf, twc, c, b, v);
        sink(i, c, b, v);
    }
    return true;
}

// Inverse transform after its first column pass; the real rows go to
// `out(y, m, off, value)` (window row y < rows, sites 2m and 2m + 1; off: where the
// value's element of the buffer was).
template <int N, int NT, class Out>
__device__ __forceinline__ void inverse_end(const Window& w, int rows, unsigned char* buf, Out out)
{
    using X = TC<N, NT>;
    const int lane = w.lane, warp = w.warp;
    __syncthreads();
#pragma unroll 1
    for (int u = warp; u < X::CA * X::CH; u += X::NW) cols8<N, true>(buf, u % X::CA, (u / X::CA) * 32 + lane);
    __syncthreads();
    // rows of the output tile only (the window's rows from `rows` on are halo)
#pragma unroll 1
    for (int u = warp; u < 4 * ((rows + 31) / 32); u += X::NW) {
        const int y = (u >> 2) * 32 + lane;
        switch (u & 3) {
            case 0: rows_inv<N, 0>(buf, y); break;
            case 1: rows_inv<N, 1>(buf, y); break;
            case 2: rows_inv<N, 2>(buf, y); break;
            default: rows_inv<N, 3>(buf, y); break;
        }
    }
    __syncthreads();
    const int m1 = lane % X::RR;
    constexpr int RPW = 32 / X::RR;
#pragma unroll 1
    for (int i = 0; i < N / (RPW * X::NW); i++) {
        const int y = (warp + i * X::NW) * RPW + lane / X::RR;
        if ((warp + i * X::NW) * RPW >= rows) break;          // warp-uniform
        const int base = y * X::PITCH + ((m1 * 8 + (m1 & 7)) ^ row_sw(y)) * 8;
        float2 v[8];
#pragma unroll
        for (int j = 0; j < 8; j++) v[j] = ld2(buf, base ^ (j * 8));
        DFT<8, true, true>::run(v);
        if (y < rows) {
#pragma unroll
            for (int m2 = 0; m2 < 8; m2++) out(y, m1 + X::RR * m2, base ^ (m2 * 8), v[m2]);
        }
    }
}

// Kernel spectrum at rows a 8 + b (a < CA) of column c.
template <int N>
__device__ __forceinline__ void spectrum_of(const float* S, int c, int b, float* s)
{
    using X = TC<N>;
    const float4* q = reinterpret_cast<const float4*>(S) + (size_t)b * (X::CA / 4) * X::M + c;
#pragma unroll
    for (int a4 = 0; a4 < X::CA / 4; a4++) {
        const float4 f = __ldg(q + (size_t)a4 * X::M);
        s[4 * a4] = f.x;
        s[4 * a4 + 1] = f.y;
        s[4 * a4 + 2] = f.z;
        s[4 * a4 + 3] = f.w;
    }
}

// Multiplies the CA spectrum values of (column c, residue b) by kernel
// spectrum S; column 0 packs the DC and Nyquist columns: f a + conj(f(-ky)) b.
template <int N>
__device__ __forceinline__ void spectral_product(const float* S, const float* S0, const float2* F0, int c, int b,
                                                 float2* v)
{
    using X = TC<N>;
    float s[X::CA];
    spectrum_of<N>(S, c, b, s);
#pragma unroll
    for (int a = 0; a < X::CA; a++) v[a] = cscale(v[a], s[a]);
    if (c == 0) {
#pragma unroll
        for (int a = 0; a < X::CA; a++) {
            const int ky = a * 8 + b;
            const float2 fm = F0[(N - ky) & (N - 1)];
            const float bb = __ldg(&S0[ky]);
            v[a].x = fmaf(fm.x, bb, v[a].x);
            v[a].y = fmaf(-fm.y, bb, v[a].y);
        }
    }
}

// Inverse transform of the spectrum that `source(i, c, b, v)` yields per task.
template <int N, int NT, int UNR, class Source, class Out>
__device__ __forceinline__ void inverse(const Window& w, int rows, unsigned char* buf, const float2* twc,
                                        Source source, Out out)
{
    using X = TC<N, NT>;
    constexpr int TASKS = 8 * X::CH / X::NW;
#pragma unroll UNR
    for (int i = 0; i < TASKS; i++) {
        const int u = w.warp + i * X::NW;
        const int b = u % 8, c = (u / 8) * 32 + w.lane;
        float2 v[X::CA];
        source(i, c, b, v);
        cols_inv<N>(buf, twc, c, b, v);
    }
    inverse_end<N, NT>(w, rows, buf, out);
}

// Whether any value of the plane `gate` within gate_r of the output tile is above
// gate_eps (whole quads of columns, so a few columns more on either side).
template <int N, int NT>
__device__ __forceinline__ bool window_live(const float* gate, const TileParams& p, const Window& w, int rows, int xend)
{
    constexpr int NW = TC<N, NT>::NW, RB = 7;
    const int nr = rows + 2 * p.gate_r, ys = w.y0 - p.gate_r;
    const int q0 = (w.x0 - p.gate_r + 4) / 4 - 1, nq = (w.x0 + xend + p.gate_r + 3) / 4 - q0;   // quads, from q0 >= -1
    bool any = false;
    for (int c = w.lane; c < nq; c += 32) {
        int x = 4 * (q0 + c);
        x = x < 0 ? x + p.W : (x >= p.W ? x % p.W : x);
        for (int r = w.warp; r < nr; r += RB * NW) {
            float4 f[RB];                                // RB rows in flight at once
#pragma unroll
            for (int j = 0; j < RB; j++) {
                const int rr = r + j * NW;
                int y = ys + rr;
                y = y < 0 ? y + p.H : (y >= p.H ? y - p.H : y);
                f[j] = rr < nr ? __ldg(reinterpret_cast<const float4*>(gate + (size_t)y * p.W + x))
                               : make_float4(p.gate_eps, p.gate_eps, p.gate_eps, p.gate_eps);
            }
#pragma unroll
            for (int j = 0; j < RB; j++)
                any |= fmaxf(fmaxf(f[j].x, f[j].y), fmaxf(f[j].z, f[j].w)) > p.gate_eps;
        }
    }
    return __syncthreads_or(any);
}

// One block: a window of channel blockIdx.y, kernels blockIdx.z kpb .. of its
// list.  ADJ: the transpose, out_c = add_c + sum_{k in list(c)} K~_k (x) plane k:
// every listed plane is transformed forward, weighted and summed in TMEM, and
// one inverse transform follows (a channel that no kernel reads gets add_c).
// With a gate (the first gene plane of a world that maintains its genes) a block
// whose output tile has no gene within the diffusion disk of any site does
// nothing: alpha is false at all of its sites, so the step never reads
// their potentials.
template <int N, int NT, bool ADJ>
__global__ void __launch_bounds__(NT, NT == 4 * N ? (N == 128 ? 2 : (ADJ ? 4 : 5)) : (N == 128 ? 3 : (ADJ ? 6 : 8)))
k_tile_conv(const __grid_constant__ TileParams p)
{
    pdl_enter();
    using X = TC<N, NT>;
    extern __shared__ __align__(128) unsigned char buf[];
    float2* F0 = reinterpret_cast<float2*>(buf + (size_t)N * X::M * 8);     // spectrum column 0 (ADJ: its mirrored sum)
    float2* twc = F0 + N;                                                    // [b][n1] w_N^(n1 b)
    __shared__ uint32_t tmem_base;
    Window w;
    w.lane = threadIdx.x & 31;
    w.warp = threadIdx.x >> 5;
    const int world = p.worlds ? (int)blockIdx.y / p.C : 0;
    w.c = p.worlds ? (int)blockIdx.y % p.C : (int)blockIdx.y;
    const TileWorld* tw = p.worlds ? p.worlds + world : nullptr;
    w.g = tw ? tw->g : p.g;
    if ((int)blockIdx.x >= w.g.tiles_x * w.g.tiles_y) return;
    const float* gA = tw ? tw->A : p.A;
    float* gU = tw ? tw->U : p.U;
    const float* gS = tw ? tw->S : p.S;
    const float* gS0 = tw ? tw->S0 : p.S0;
    const int nk = !ADJ && p.per_plane ? 1 : p.kcount[w.c];
    const int t0 = ADJ ? 0 : (int)blockIdx.z * p.kpb;
    if (!ADJ && t0 >= nk) return;                                            // uniform over the block
    const int t1 = ADJ ? nk : min(nk, t0 + p.kpb);
    w.x0 = (int)(blockIdx.x % w.g.tiles_x) * w.g.vx;
    w.y0 = (int)(blockIdx.x / w.g.tiles_x) * w.g.vy;
    const size_t HW = (size_t)p.H * p.W;
    const int rows = min(w.g.vy, p.H - w.y0);
    const int xend = min(w.g.vx, p.W - w.x0);
    if constexpr (!ADJ) {
        if (p.gate && !window_live<N, NT>(p.gate, p, w, rows, xend)) return;
    } else if (nk == 0) {
        // a channel that no kernel reads: its sum is empty
        for (int i = threadIdx.x; i < rows * xend; i += X::T) {
            const size_t o = (size_t)w.c * HW + (size_t)(w.y0 + i / xend) * p.W + w.x0 + i % xend;
            gU[o] = p.add ? __ldg(p.add + o) : 0.f;
        }
        return;
    }
    if (w.warp == 0) {
        tmem_alloc<X::TMEM>(&tmem_base);
        tmem_fence_before_sync();
    }
    for (int i = threadIdx.x; i < N; i += X::T) twc[i] = __ldg(&p.tw[i]);
    if (ADJ)
        for (int i = threadIdx.x; i < N; i += X::T) F0[i] = make_float2(0.f, 0.f);
    __syncthreads();
    tmem_fence_after_sync();
    constexpr int FPT = 2 * X::CA;                                           // floats per task
    constexpr int TASKS = 8 * X::CH / X::NW;
    // both tasks of a thread in flight, where that needs no spills
    constexpr int UNR = ADJ && N == 128 ? 1 : TASKS;
    const uint32_t taddr = tmem_base + ((uint32_t)(32 * (w.warp & 3)) << 16) +
                           (uint32_t)((w.warp >> 2) * (FPT * TASKS));
    auto tput = [&](int i, const float2* v) {
        const float* f = reinterpret_cast<const float*>(v);
        tmem_st16(taddr + i * FPT, f);
        if constexpr (FPT == 32) tmem_st16(taddr + i * FPT + 16, f + 16);
    };
    auto tget = [&](int i, float2* v) {
        float* f = reinterpret_cast<float*>(v);
        tmem_ld16(taddr + i * FPT, f);
        if constexpr (FPT == 32) tmem_ld16(taddr + i * FPT + 16, f + 16);
    };
    const size_t SP = (size_t)N * X::M;                                      // floats of one kernel spectrum
    if constexpr (!ADJ) {
        const float* plane = gA + (size_t)w.c * HW;
        const bool usual = forward<N, NT, UNR>(p, plane, w, buf, twc, [&](int i, int c, int b, float2* v) {
            tput(i, v);
            if (c == 0)
#pragma unroll
                for (int a = 0; a < X::CA; a++) F0[a * 8 + b] = v[a];
        });
        tmem_wait_st();
        __syncthreads();
        if (!usual) window_direct<false>(p, w.c, t0, t1, w.x0, w.y0, rows, xend);
        else
        for (int t = t0; t < t1; t++) {
            const int k = p.per_plane ? w.c : p.klist[w.c][t];
            float* U = gU + (size_t)k * HW;
            inverse<N, NT, UNR>(
                w, rows, buf, twc,
                [&](int i, int c, int b, float2* v) {
                    tget(i, v);
                    spectral_product<N>(gS + (size_t)k * SP, gS0 + (size_t)k * N, F0, c, b, v);
                },
                [&](int y, int m, int, float2 v) {
                    if (2 * m < xend) {
                        float* o = U + (size_t)(w.y0 + y) * p.W + w.x0 + 2 * m;
                        if (p.vec2o) *reinterpret_cast<float2*>(o) = v;
                        else {
                            o[0] = v.x;
                            o[1] = v.y;
                        }
                    }
                });
            __syncthreads();
        }
    } else {
        bool usual = true;
        for (int t = 0; usual && t < nk; t++) {
            const int k = p.klist[w.c][t];
            usual = forward<N, NT, UNR>(p, gA + (size_t)k * HW, w, buf, twc, [&](int i, int c, int b, float2* v) {
                if (c == 0) {
                    // mirrored share of the packed column, at -ky (this thread's slots only)
                    const float* s2 = gS0 + (size_t)k * N;
#pragma unroll
                    for (int a = 0; a < X::CA; a++) {
                        const int ky = a * 8 + b, kn = (N - ky) & (N - 1);
                        const float bb = __ldg(&s2[ky]);
                        F0[kn] = make_float2(fmaf(v[a].x, bb, F0[kn].x), fmaf(-v[a].y, bb, F0[kn].y));
                    }
                }
                float s[X::CA];
                spectrum_of<N>(gS + (size_t)k * SP, c, b, s);
                float2 acc[X::CA];
                if (t > 0) tget(i, acc);
#pragma unroll
                for (int a = 0; a < X::CA; a++) {
                    v[a] = cscale(v[a], s[a]);
                    if (t > 0) v[a] = cadd(acc[a], v[a]);
                }
                tput(i, v);
            });
            tmem_wait_st();
            __syncthreads();
        }
        float* O = gU + (size_t)w.c * HW;
        const float* add = p.add ? p.add + (size_t)w.c * HW : nullptr;
        if (!usual) window_direct<true>(p, w.c, 0, nk, w.x0, w.y0, rows, xend);
        else
        inverse<N, NT, UNR>(
            w, rows, buf, twc,
            [&](int i, int c, int b, float2* v) {
                tget(i, v);
                if (c == 0)
#pragma unroll
                    for (int a = 0; a < X::CA; a++) v[a] = cadd(v[a], F0[a * 8 + b]);
            },
            [&](int y, int m, int, float2 v) {
                if (2 * m < xend) {
                    const size_t o = (size_t)(w.y0 + y) * p.W + w.x0 + 2 * m;
                    if (add) {
                        v.x = __ldg(add + o) + v.x;
                        v.y = __ldg(add + o + 1) + v.y;
                    }
                    if (p.vec2o) *reinterpret_cast<float2*>(O + o) = v;
                    else {
                        O[o] = v.x;
                        O[o + 1] = v.y;
                    }
                }
            });
    }
    tmem_fence_before_sync();
    __syncthreads();
    if (w.warp == 0) {
        tmem_fence_after_sync();
        tmem_dealloc<X::TMEM>(tmem_base);
    }
}

// A whole rollout of a one-channel world with global genes whose torus is one
// window (64^2 or 128^2): one block, every step in shared memory and registers.
// A thread holds the same eight pairs of sites of its rows through the whole
// rollout: they are what its last inverse pass yields and its first forward
// pass takes, so a step is the seven in-place passes above with a barrier after
// each, the growth in registers, and nothing in global memory.  What bounds it
// is the latency of those passes (64^2, one kernel: see the launch's comment).
template <int N, bool ONE>
__host__ __device__ constexpr bool rollout_stash() { return N == 128 && !ONE; }
template <int N, bool ONE>
__global__ void __launch_bounds__(4 * N, 1) k_tile_rollout(const __grid_constant__ TileRolloutParams p)
{
    pdl_enter();
    using X = TC<N>;
    constexpr int T = 4 * N, NW = T / 32, RPW = 32 / X::RR, NR = N / (RPW * NW);
    extern __shared__ __align__(128) unsigned char buf[];
    float2* F0 = reinterpret_cast<float2*>(buf + (size_t)N * X::M * 8);
    float2* twc = F0 + N;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int m1 = lane % X::RR;
    for (int i = threadIdx.x; i < N; i += T) twc[i] = __ldg(&p.tw[i]);
    int ys[NR], base[NR];
    // The state: rows ys[i], pairs m1 + RR m2.  Several kernels of 128^2: beside the growth's
    // sums neither it nor the spectrum fits the registers; it waits in shared memory,
    // the spectrum in TMEM (each thread's share in its own lane).
    constexpr bool TM = rollout_stash<N, ONE>();
    float2 a[TM ? 1 : NR][8];
    float2* stash = twc + N + threadIdx.x;
    auto state = [&](int i, int j) -> float2& {
        if constexpr (TM) return stash[(i * 8 + j) * T];
        else return a[i][j];
    };
    __shared__ uint32_t tmem_base;
    if (TM && warp == 0) {
        tmem_alloc<TM ? X::TMEM : 32>(&tmem_base);
        tmem_fence_before_sync();
    }
#pragma unroll
    for (int i = 0; i < NR; i++) {
        ys[i] = (warp + i * NW) * RPW + lane / X::RR;
        base[i] = ys[i] * X::PITCH + ((m1 * 8 + (m1 & 7)) ^ row_sw(ys[i])) * 8;
#pragma unroll
        for (int m2 = 0; m2 < 8; m2++) {
            const float* q = p.A + (size_t)ys[i] * N + 2 * (m1 + X::RR * m2);
            state(i, m2) = make_float2(q[0], q[1]);
        }
    }
    // this thread's column task, one per thread
    static_assert(8 * X::CH == NW, "one column task per thread");
    const int b = warp % 8, c = (warp / 8) * 32 + lane;
    float s1[X::CA];
    if (ONE) spectrum_of<N>(p.S, c, b, s1);
    __syncthreads();
    if (TM) tmem_fence_after_sync();
    const uint32_t taddr = TM ? tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * 2 * X::CA) : 0;
    for (int t = 0; t < p.n_steps; t++) {
#pragma unroll
        for (int i = 0; i < NR; i++) {
            float2 v[8];
#pragma unroll
            for (int m2 = 0; m2 < 8; m2++) v[m2] = state(i, m2);
            DFT<8, false, true>::run(v);
#pragma unroll
            for (int j = 0; j < 8; j++) st2(buf, base[i] ^ (j * 8), v[j]);
        }
        __syncthreads();
        for (int u = warp; u < 4 * (N / 32); u += NW) {
            const int y = (u >> 2) * 32 + lane;
            switch (u & 3) {
                case 0: rows_fwd<N, 0>(buf, y); break;
                case 1: rows_fwd<N, 1>(buf, y); break;
                case 2: rows_fwd<N, 2>(buf, y); break;
                default: rows_fwd<N, 3>(buf, y); break;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = warp; u < X::CA * X::CH; u += NW) cols8<N, false>(buf, u % X::CA, (u / X::CA) * 32 + lane);
        __syncthreads();
        float2 f[X::CA];
        cols_fwd<N>(buf, twc, c, b, f);
        if (c == 0) {
#pragma unroll
            for (int i = 0; i < X::CA; i++) F0[i * 8 + b] = f[i];
        }
        if constexpr (TM) {
            const float* w = reinterpret_cast<const float*>(f);
            tmem_st16(taddr, w);
            tmem_st16(taddr + 16, w + 16);
            tmem_wait_st();
        }
        float2 acc[NR][8];
        for (int k = 0; k < (ONE ? 1 : p.K); k++) {
            __syncthreads();                             // F0 complete; the last kernel's rows are read
            float2 v[X::CA];
#pragma unroll
            for (int i = 0; i < X::CA; i++) v[i] = f[i];
            if constexpr (TM) {
                float* w = reinterpret_cast<float*>(v);
                tmem_ld16(taddr, w);
                tmem_ld16(taddr + 16, w + 16);
            }
            if (ONE && c != 0) {
#pragma unroll
                for (int i = 0; i < X::CA; i++) v[i] = cscale(v[i], s1[i]);
            } else {
                spectral_product<N>(p.S + (size_t)k * N * X::M, p.S0 + (size_t)k * N, F0, c, b, v);
            }
            cols_inv<N>(buf, twc, c, b, v);
            __syncthreads();
#pragma unroll
            for (int u = warp; u < X::CA * X::CH; u += NW) cols8<N, true>(buf, u % X::CA, (u / X::CA) * 32 + lane);
            __syncthreads();
            for (int u = warp; u < 4 * (N / 32); u += NW) {
                const int y = (u >> 2) * 32 + lane;
                switch (u & 3) {
                    case 0: rows_inv<N, 0>(buf, y); break;
                    case 1: rows_inv<N, 1>(buf, y); break;
                    case 2: rows_inv<N, 2>(buf, y); break;
                    default: rows_inv<N, 3>(buf, y); break;
                }
            }
            __syncthreads();
            const float m = p.mu[k], sg = p.sigma[k], rs = p.rsigma[k], h = p.h[k];
            // (u - m) / sigma by the reciprocal and one residual correction, and expf: with
            // the quotient uncorrected and the hardware exponential the errors of 24 rollouts
            // (64^2, 16 steps) had a geometric mean of 8.9e-7 and a largest of 4.0e-6; with
            // IEEE division 8.6e-7 and 2.5e-6, which a step 20% longer paid for
            auto growth = [&](float u) {
                const float d = u - m, q = d * rs;
                const float z = fmaf(fmaf(-q, sg, d), rs, q);
                const float g = expf(-0.5f * z * z);
                return p.growth_form == 0 ? h * fmaf(2.f, g, -1.f) : h * g;
            };
#pragma unroll
            for (int i = 0; i < NR; i++) {
#pragma unroll
                for (int j = 0; j < 8; j++) v[j] = ld2(buf, base[i] ^ (j * 8));
                DFT<8, true, true>::run(v);
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const float2 g = make_float2(growth(v[j].x), growth(v[j].y));
                    acc[i][j] = k == 0 ? g : make_float2(acc[i][j].x + g.x, acc[i][j].y + g.y);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NR; i++)
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const float2 s = state(i, j);
                state(i, j) = make_float2(__saturatef(fmaf(p.dt, acc[i][j].x, s.x)), __saturatef(fmaf(p.dt, acc[i][j].y, s.y)));
            }
    }
#pragma unroll
    for (int i = 0; i < NR; i++)
#pragma unroll
        for (int m2 = 0; m2 < 8; m2++) {
            float* q = p.A + (size_t)ys[i] * N + 2 * (m1 + X::RR * m2);
            q[0] = state(i, m2).x;
            q[1] = state(i, m2).y;
        }
    if (TM) {
        tmem_fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            tmem_fence_after_sync();
            tmem_dealloc<TM ? X::TMEM : 32>(tmem_base);
        }
    }
}

// Kernel spectra in the order the column tasks read them, from S[kx][ky] of the
// N x N torus (kx, ky in 0..N/2): row ky = a 8 + b of column c goes to
// [b][a / 4][c][a % 4]; the factor 1/2 undoes the doubled forward spectrum.
// Column 0 keeps (s0 + sN) / 2 here and (s0 - sN) / 2 in S0.
template <int N>
__global__ void k_tile_spectra(const float* S, float* out, float* out0)
{
    constexpr int M = N / 2, HS = N / 2 + 1, CA = N / 8;
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= N * M) return;
    const int ky = u / M, c = u % M;
    const int a = ky / 8, b = ky % 8, kyr = ky <= N / 2 ? ky : N - ky;
    float v = S[c * HS + kyr];
    if (c == 0) {
        const float sn = S[M * HS + kyr];
        out0[ky] = 0.25f * (v - sn);
        v = 0.5f * (v + sn);
    }
    out[(((size_t)b * (CA / 4) + a / 4) * M + c) * 4 + a % 4] = 0.5f * v;
}

// Blocks of one window and one share of a channel's kernels.
dim3 conv_grid(const TileParams& p, bool adj)
{
    int kmax = p.per_plane ? 1 : 0;
    for (int c = 0; c < p.C && c < kMaxChannels && !p.per_plane; c++) kmax = p.kcount[c] > kmax ? p.kcount[c] : kmax;
    return dim3(p.worlds ? p.tiles : p.g.tiles_x * p.g.tiles_y, p.worlds ? p.C * p.n_worlds : p.C,
                adj ? (kmax > 0) : (kmax + p.kpb - 1) / p.kpb);
}

template <int N, int NT, bool ADJ>
cudaError_t launch_nt(const TileParams& p, const dim3& grid, cudaStream_t s)
{
    cudaError_t e = smem_limit<k_tile_conv<N, NT, ADJ>>(TC<N, NT>::SMEM);
    if (e != cudaSuccess) return e;
    launch_pdl(k_tile_conv<N, NT, ADJ>, grid, NT, TC<N, NT>::SMEM, s, p);
    return cudaGetLastError();
}

// Threads of a block.  Each pass has the same tasks with either count, so the
// values do not depend on it.  With few blocks the SMs are short of warps and
// 4 N threads are faster; with many, 2 N keep more windows in flight and spare
// registers.  Measured (us, 2 N against 4 N threads; R = 18 unless stated):
//   N = 64   one window 5.8 / 4.8, 300 x 404 6.5 / 5.5, 256^2 15 kernels in 147
//            blocks 15.9 / 14.4, in 245 12.9 / 12.4, in 390 12.4 / 12.6, in 735
//            13.6 / 14.6, 1080 x 1920 15 kernels 131 / 143
//   N = 128  256^2 15 kernels in 135 blocks 12.6 / 11.0, 1024^2 one kernel (121
//            blocks) 11.8 / 10.4, 2048^2 one kernel (441) 23.1 / 24.0, 15 kernels
//            190 / 196
// hence the line at two blocks an SM.  Where a gate skips windows the blocks
// that work are few again (N = 128, 1080 x 1920 15 kernels, a quarter live:
// 66 / 52; 2048^2, 28% live: 112 / 106).  The transposed sum of N = 128 would
// spill at 4 N threads.
bool wide_block(int N, int n_sms, double blocks, bool gated, bool adj)
{
    if (N == 128 && adj) return false;
    return blocks <= 2.0 * n_sms || (N == 128 && gated);
}

template <int N, bool ADJ>
cudaError_t launch_n(const TileParams& p, cudaStream_t s)
{
    const dim3 grid = conv_grid(p, ADJ);
    if (grid.z == 0) return cudaSuccess;
    if constexpr (!(N == 128 && ADJ)) {
        if (wide_block(N, p.n_sms, (double)grid.x * grid.y * grid.z, p.gate != nullptr, ADJ)) return launch_nt<N, 4 * N, ADJ>(p, grid, s);
    }
    return launch_nt<N, 2 * N, ADJ>(p, grid, s);
}

}  // namespace

size_t tile_spectrum_floats(int N) { return (size_t)N * (N / 2); }

cudaError_t launch_tile_spectra(int N, const float* S, float* out, float* out0, cudaStream_t s)
{
    const int n = N * (N / 2);
    if (N == 128) k_tile_spectra<128><<<(n + 255) / 256, 256, 0, s>>>(S, out, out0);
    else k_tile_spectra<64><<<(n + 255) / 256, 256, 0, s>>>(S, out, out0);
    return cudaGetLastError();
}

bool tile_plan(TileParams* p, int N, int H, int W, int R)
{
    if (N != 64 && N != 128) return false;
    p->N = N;
    p->H = H;
    p->W = W;
    // pairs of columns travel together, so the halo along x is even
    const int Rx = (R + 1) / 2 * 2;
    p->g.vx = W == N ? N : N - 2 * Rx;
    p->g.vy = H == N ? N : N - 2 * R;
    if (p->g.vx < 16 || p->g.vy < 16) return false;
    p->g.halo_x = W == N ? 0 : Rx;
    p->g.halo_y = H == N ? 0 : R;
    p->g.cut_x = p->g.vx + p->g.halo_x;
    p->g.cut_y = p->g.vy + p->g.halo_y;
    p->g.tiles_x = (W + p->g.vx - 1) / p->g.vx;
    p->g.tiles_y = (H + p->g.vy - 1) / p->g.vy;
    return true;
}

// Time model of one launch (us), fitted to measurements at 64^2 .. 2048^2: a
// block's work is two units for the forward transform and one per kernel; a
// unit takes t1 on an idle SM and tf with every block slot of the SM taken.
static double tile_time(const TileParams& p, double blocks, double units, bool adj)
{
    const bool wide = wide_block(p.N, p.n_sms, blocks, false, adj);
    const double slots = (double)p.n_sms * (wide ? 2 : p.N == 128 ? 3 : 8);
    const double t1 = p.N == 128 ? (wide ? 2.0 : 2.3) : wide ? 0.6 : 0.9;
    const double tf = p.N == 128 ? (wide ? 3.8 : 7.7) : wide ? 2.2 : 4.2;
    const double waves = blocks / slots, whole = floor(waves), rest = waves - whole;
    return 3.0 + units * (whole * tf + (rest > 0 ? t1 + (tf - t1) * rest : 0));
}

static double tile_cost(const TileParams& p, const int* kcount, int kpb, int n_worlds)
{
    double blocks = 0;
    int kmax = 0;
    for (int c = 0; c < kMaxChannels; c++) {
        blocks += (double)n_worlds * p.g.tiles_x * p.g.tiles_y * ((kcount[c] + kpb - 1) / kpb);
        kmax = kcount[c] > kmax ? kcount[c] : kmax;
    }
    return tile_time(p, blocks, 2 + (kpb < kmax ? kpb : kmax), false);
}

double tile_adj_cost(const TileParams& p, const int* kcount)
{
    int kmax = 0, chans = 0;
    for (int c = 0; c < kMaxChannels; c++) {
        kmax = kcount[c] > kmax ? kcount[c] : kmax;
        chans += kcount[c] > 0;
    }
    return tile_time(p, (double)p.g.tiles_x * p.g.tiles_y * chans, 1 + 2 * kmax, true);
}

double tile_planes_cost(const TileParams& p, int K)
{
    return tile_time(p, (double)p.g.tiles_x * p.g.tiles_y * K, 3, false);
}

double tile_choose(TileParams* p, int H, int W, const int* kcount, int R, int n_worlds, bool gated)
{
    double best = INFINITY;
    int kmax = 0;
    for (int c = 0; c < kMaxChannels; c++) kmax = kcount[c] > kmax ? kcount[c] : kmax;
    for (int N : {64, 128}) {
        TileParams q = *p;
        if (!tile_plan(&q, N, H, W, R)) continue;
        for (int kpb = 1; kpb <= kmax; kpb++) {
            const double t = tile_cost(q, kcount, kpb, n_worlds);
            // near ties go to the larger window where a gate may skip some (its check is
            // the smaller part of a window's work: 2048^2, 15 kernels R = 5, a
            // quarter live: 87 against 97 us)
            if (t >= (gated && N == 128 && p->N == 64 ? 1.08 * best : best)) continue;
            best = t;
            *p = q;
            p->kpb = kpb;
        }
    }
    return best;
}

void tile_choose_kpb(TileParams* p, const int* kcount, int n_worlds)
{
    int kmax = 0;
    for (int c = 0; c < kMaxChannels; c++) kmax = kcount[c] > kmax ? kcount[c] : kmax;
    double best = INFINITY;
    for (int kpb = 1; kpb <= kmax; kpb++) {
        const double t = tile_cost(*p, kcount, kpb, n_worlds);
        if (t >= best) continue;
        best = t;
        p->kpb = kpb;
    }
}

double fft_passes_cost(int H, int W, int planes) { return 9.0 + 2.6e-6 * H * W * planes; }

double direct_cost(int H, int W, int planes, int R)
{
    const double taps = 3.1416 * R * R;
    return 4.0 + fmax(taps * H * W * planes / 14.0e6, 0.035 * taps);
}

cudaError_t launch_tile_conv(const TileParams& p0, cudaStream_t s)
{
    TileParams p = p0;
    p.vec2 = p.worlds ? p.aligned : ((uintptr_t)p.A & 7) == 0;
    p.vec2o = p.worlds ? p.aligned : ((uintptr_t)p.U & 7) == 0;
    return p.N == 128 ? launch_n<128, false>(p, s) : launch_n<64, false>(p, s);
}

// Where one block pays (us for 2 / 6 / 16 steps against the same steps as launches):
//   64^2   one kernel 8 / 13 / 30 against 17 / 56 / 148, four 14 / 34 / 86 against 17 /
//          50 / 132
//   128^2  one kernel 18 / 45 / 112 against 17 / 50 / 132, three (from four steps on) 99 /
//          255 against 56 / 148 (99 / 263 with the FFT passes)
int tile_rollout_steps(int H, int W, int C, int K)
{
    if (H != W || C != 1) return 0;
    if (H == 64) return K <= kTileRolloutKernels ? 2 : 0;
    return H == 128 && K <= 3 ? (K == 1 ? 2 : 4) : 0;
}

template <int N, bool ONE>
static cudaError_t launch_rollout_n(const TileRolloutParams& p, cudaStream_t s)
{
    const size_t smem = TC<N>::SMEM + (rollout_stash<N, ONE>() ? (size_t)N * N * sizeof(float) : 0);
    cudaError_t e = smem_limit<k_tile_rollout<N, ONE>>(smem);
    if (e != cudaSuccess) return e;
    launch_pdl(k_tile_rollout<N, ONE>, dim3(1), dim3(4 * N), smem, s, p);
    return cudaGetLastError();
}

cudaError_t launch_tile_rollout(const TileRolloutParams& p, int N, cudaStream_t s)
{
    if (N == 64) return p.K == 1 ? launch_rollout_n<64, true>(p, s) : launch_rollout_n<64, false>(p, s);
    return p.K == 1 ? launch_rollout_n<128, true>(p, s) : launch_rollout_n<128, false>(p, s);
}

cudaError_t launch_tile_conv_adj(const TileParams& p0, cudaStream_t s)
{
    TileParams p = p0;
    p.vec2 = ((uintptr_t)p.A & 7) == 0;
    p.vec2o = ((uintptr_t)p.U & 7) == 0;
    return p.N == 128 ? launch_n<128, true>(p, s) : launch_n<64, true>(p, s);
}

}  // namespace lenia

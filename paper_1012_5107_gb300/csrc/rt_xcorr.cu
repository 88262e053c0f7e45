// rt_xcorr.cu -- image cross-correlation C(0,0) of Eqs. 14-15 (Sec. 5).
//
// The window sums are moments (sum f, sum g, sum f^2, sum f g) per channel in
// FP64 or better.  FP64 arithmetic is slow on this GPU (two fused
// multiply-adds per SM and cycle: six operations a value made it the bound),
// so the first pass sums in three floats with error-free transformations on the
// FP32 pipe (two floats are not enough: photographs repeat their values, and the
// rounding of a value's low part adds up), and only its results are FP64:
//   1. a block takes 32 columns of the flattened row at a time (one per lane, so
//      loads are coalesced) and splits its row chunk over its 8 warps; from the
//      32 columns' moments it adds those of each window and channel.  The
//      chunks are as many as give two blocks an SM, and a block goes on to
//      further columns where there are more than that;
//   2. a block per window adds the blocks' moments and forms
//        C_c = (S_fg - S_f S_g / N) / (S_ff - S_f^2 / N)
//      per channel (the numerator and denominator of Eq. 15 after the mean
//      subtraction of Eq. 14) and the same ratio over the stacked channels.
// Images of at most 4096 values and 64 values per row (a centre line) take
// one block instead: a launch costs more than their arithmetic.
// The order of the additions is fixed, so results repeat bit for bit.
//
// Measured: a 512 x 512 x 3 pair at three fields of view and its centre lines,
// as a program issues them, 48 us -> 27 us (54 us instead of 285 us when it
// waits for each), of which the full frame 15 us and a centre line 7 us on the
// GPU.  What is left of the frame is two dependent launches over 6 MB.  Against
// 64 bits C is 3.8e-15 off (7.6e-15 with FP64 moments; geometric means over 40
// sizes and inputs, single frames from 1e-15 to 3e-14).
#include <algorithm>
#include <cmath>

#include "rt_internal.h"
#include "rt_moments.cuh"

namespace grt {

constexpr int kXcorrBlock = 256;
constexpr int kXcorrWarps = kXcorrBlock / 32;
constexpr int kXcorrBlocks = 304;      // blocks wanted in pass 1 (two per SM)
constexpr int kXcorrSmallRow = 64;     // one-block path: values per row (W C) at most
constexpr int kXcorrSmallAll = 4096;   // and values (H W C) at most
static_assert(kXcorrScratch >= (size_t)2 * kXcorrBlocks * kMaxWindows * 16 * sizeof(double), "scratch too small");

// Grid of pass 1: column tiles (at most kXcorrBlocks) x row chunks (at most
// one per 8 rows, a row per warp; less than 2 kXcorrBlocks in all).
static dim3 xcorr_grid(int H, int W, int C)
{
    const int64_t tiles = std::min<int64_t>(((int64_t)W * C + 31) / 32, kXcorrBlocks);
    const int64_t chunks = std::min<int64_t>((kXcorrBlocks + tiles - 1) / tiles, ((int64_t)H + kXcorrWarps - 1) / kXcorrWarps);
    return dim3((unsigned)tiles, (unsigned)chunks);
}

static bool xcorr_one_block(int H, int W, int C)
{
    const int64_t WC = (int64_t)W * C;
    return WC <= kXcorrSmallRow && (int64_t)H * WC <= kXcorrSmallAll;
}

size_t xcorr_scratch_bytes(int H, int W, int C, int n_fov)
{
    if (xcorr_one_block(H, W, C)) return 0;
    const dim3 g = xcorr_grid(H, W, C);
    return (size_t)g.x * g.y * (size_t)n_fov * 4 * C * sizeof(double);
}

// Moments of 32 columns over the block's rows, to col[moment][column] (threads
// 0..63 write them; the caller synchronises).  A tile with a value outside
// xcorr_plain is summed in FP64, as all were.
__device__ __forceinline__ void xcorr_tile(const float* __restrict__ f, const float* __restrict__ g, int WC, int q0,
                                           int i0, int i1, Z3 (*red3)[kXcorrWarps][32], double (*col)[32])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = q0 + lane;
    Z3 s1 = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, s2 = s1;   // (f, g) and (f^2, f g)
    int odd = 0;
    if (q < WC) {
#pragma unroll 4
        for (int i = i0 + warp; i < i1; i += kXcorrWarps) {
            const float a = __ldg(f + (size_t)i * WC + q), b = __ldg(g + (size_t)i * WC + q);
            odd |= !(xcorr_plain(a) && xcorr_plain(b));
            const F2 p = two_prod(a, a), r = two_prod(a, b);
            xcorr_add(s1, float2{a, b});
            xcorr_add(s2, float2{p.h, r.h});
            xcorr_low(s2, float2{p.l, r.l});
        }
    }
    if (__syncthreads_or(odd)) {
        double(*red)[kXcorrWarps][32] = reinterpret_cast<double(*)[kXcorrWarps][32]>(red3);
        double sf = 0.0, sg = 0.0, sff = 0.0, sfg = 0.0;
        if (q < WC) {
            for (int i = i0 + warp; i < i1; i += kXcorrWarps) {
                const double a = __ldg(f + (size_t)i * WC + q), b = __ldg(g + (size_t)i * WC + q);
                sf += a;
                sg += b;
                sff += a * a;
                sfg += a * b;
            }
        }
        red[0][warp][lane] = sf;
        red[1][warp][lane] = sg;
        red[2][warp][lane] = sff;
        red[3][warp][lane] = sfg;
        __syncthreads();
        if (threadIdx.x < 2 * 32)
            for (int m = 2 * warp; m < 2 * warp + 2; ++m) {
                double s = 0.0;
#pragma unroll
                for (int w = 0; w < kXcorrWarps; ++w) s += red[m][w][lane];
                col[m][lane] = s;
            }
        return;
    }
    red3[0][warp][lane] = s1;
    red3[1][warp][lane] = s2;
    __syncthreads();
    if (threadIdx.x < 2 * 32) {
        Z3 s = red3[warp][0][lane];
#pragma unroll
        for (int w = 1; w < kXcorrWarps; ++w) {
            const Z3 v = red3[warp][w][lane];
            xcorr_add(s, v.h);
            xcorr_low(s, v.m);
            s.l = vadd(s.l, v.l);
        }
        col[2 * warp][lane] = join_x(s);
        col[2 * warp + 1][lane] = join_y(s);
    }
}

// Thread o < n_win 4 C adds the moment (window, channel, m), o = (w C + c) 4 + m,
// of the block's columns; sums[w][block][4 c + m].
static_assert(kMaxWindows * 16 <= kXcorrBlock, "one thread per window and value");
__global__ void __launch_bounds__(kXcorrBlock) xcorr_moments(const float* __restrict__ f, const float* __restrict__ g,
                                                           int H, int W, int C, int rows_per_chunk, Windows win,
                                                           double* __restrict__ sums)
{
    __shared__ Z3 red3[2][kXcorrWarps][32];               // moments 0 and 1 (2 and 3) of a column as one pair
    __shared__ double col[4][32];
    static_assert(sizeof(red3) >= 4 * kXcorrWarps * 32 * sizeof(double), "the FP64 view of the sums");
    const int WC = W * C, V = 4 * C;
    const int i0 = blockIdx.y * rows_per_chunk, i1 = min(H, i0 + rows_per_chunk);
    const int t = threadIdx.x;
    const int w = t / V, c = (t - w * V) >> 2, m = t & 3;         // V is a multiple of 4
    const bool mine = w < win.n;
    const int j0 = mine ? win.j0[w] : 0, j1 = mine ? win.j1[w] : 0;
    double acc = 0.0;
    // (counted in tiles: q0 would pass 2^31 behind a row that nearly fills it)
    const int tiles = (int)(((int64_t)WC + 31) / 32);
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int q0 = tile * 32;
        xcorr_tile(f, g, WC, q0, i0, i1, red3, col);
        __syncthreads();
        // the tile's columns of channel c: pixels (q0 + l) / C, l = first, first + C, ...
        const int first = (c + C - q0 % C) % C;
        int j = (q0 + first) / C;
        for (int l = first; l < 32; l += C, ++j)
            if (j >= j0 && j < j1) acc += col[m][l];
    }
    if (mine) sums[((size_t)w * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x) * V + (t - w * V)] = acc;
}

// C of a window by eight lanes of a warp, lane c of them holding channel c's
// moments m[4] (c < C): per channel, and over the stacked channels on lane C.
// Every lane divides at the same time: FP64 divisions one after another in one
// thread took more than the sums.
__device__ __forceinline__ void xcorr_form(const double m[4], double N, int c, int C, double* __restrict__ out)
{
    const unsigned group = 0xffu << (threadIdx.x & 24u);
    const double num = c < C ? m[3] - m[0] * m[1] / N : 0.0;
    const double den = c < C ? m[2] - m[0] * m[0] / N : 0.0;
    double num_all = 0.0, den_all = 0.0;
    for (int k = 0; k < C; ++k) {
        num_all += __shfl_sync(group, num, k, 8);
        den_all += __shfl_sync(group, den, k, 8);
    }
    if (c <= C) out[c] = (c < C ? num : num_all) / (c < C ? den : den_all);
}

// Pass 2: block w adds the nb blocks' moments of its window, T threads with T a
// multiple of V = 4 C, so that each meets one of the V values; then two rounds
// over the threads of a value.
__global__ void __launch_bounds__(kXcorrBlock) xcorr_windows(const double* __restrict__ sums, int nb, int H, int C,
                                                           Windows win, double* __restrict__ out)
{
    __shared__ double red[kXcorrBlock];
    constexpr int kWays = 8;
    const int w = blockIdx.x, t = threadIdx.x, V = 4 * C;
    const int T = (kXcorrBlock / V) * V;
    double acc = 0.0;
    if (t < T) {
#pragma unroll 8
        for (int k = t; k < nb * V; k += T) acc += __ldg(sums + (size_t)w * nb * V + k);
    }
    red[t] = acc;
    __syncthreads();
    double v = 0.0;
    if (t < kWays * V)
        for (int k = t; k < T; k += kWays * V) v += red[k];
    __syncthreads();
    red[t] = v;
    __syncthreads();
    if (t >= 8) return;
    double m[4];
    for (int k = 0; k < 4; ++k) {
        double s = 0.0;
#pragma unroll
        for (int r = 0; r < kWays; ++r) s += t < C ? red[r * V + 4 * t + k] : 0.0;
        m[k] = s;
    }
    xcorr_form(m, (double)H * (double)max(0, win.j1[w] - win.j0[w]), t, C, out + w * (C + 1));
}

// The one-block path.  Threads stride over the image's values with a
// stride T that is a multiple of W C, so each meets one column and channel
// (q = t mod W C); the column moments are the sums over the threads of each
// q, and one thread per window adds its columns and forms C as in pass 3.
__global__ void __launch_bounds__(kXcorrBlock) xcorr_small(const float* __restrict__ f, const float* __restrict__ g,
                                                         int H, int W, int C, Windows win, double* __restrict__ out)
{
    __shared__ double red[4][kXcorrBlock];
    __shared__ double col[4][kXcorrSmallRow];
    const int WC = W * C;
    const int T = (kXcorrBlock / WC) * WC;
    const int n = H * WC;
    const int t = threadIdx.x;
    double sf = 0.0, sg = 0.0, sff = 0.0, sfg = 0.0;
    if (t < T) {
#pragma unroll 4
        for (int e = t; e < n; e += T) {
            const double a = __ldg(f + e), b = __ldg(g + e);
            sf += a;
            sg += b;
            sff += a * a;
            sfg += a * b;
        }
    }
    red[0][t] = sf;
    red[1][t] = sg;
    red[2][t] = sff;
    red[3][t] = sfg;
    __syncthreads();
    // the threads of a column in two rounds, `ways` partial sums first: one
    // round of T / W C additions (85 for a centre line) was most of the kernel
    const int ways = min(16, max(1, kXcorrBlock / (4 * WC)));
    double part = 0.0;
    const int item = t / ways, m = item / WC, q = item - m * WC;
    if (item < 4 * WC)
        for (int k = q + (t - item * ways) * WC; k < T; k += ways * WC) part += red[m][k];
    __syncthreads();
    red[0][t] = part;
    __syncthreads();
    for (int k = t; k < 4 * WC; k += kXcorrBlock) {
        double acc = 0.0;
        for (int r = 0; r < ways; ++r) acc += red[0][k * ways + r];
        col[k / WC][k % WC] = acc;
    }
    __syncthreads();
    // eight threads per window, one of them per channel
    const int w = t >> 3, c = t & 7;
    if (w >= win.n) return;
    const int j0 = win.j0[w], j1 = win.j1[w];
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (c < C)
        for (int j = j0; j < j1; ++j)
            for (int k = 0; k < 4; ++k) v[k] += col[k][j * C + c];
    xcorr_form(v, (double)H * (double)max(0, j1 - j0), c, C, out + w * (C + 1));
}
static_assert(8 * kMaxWindows <= kXcorrBlock, "eight finishing threads per window");

cudaError_t launch_xcorr(const float* f, const float* g, int H, int W, int C, const Windows& win, void* scratch,
                         double* out, cudaStream_t stream)
{
    if (xcorr_one_block(H, W, C)) {
        xcorr_small<<<1, kXcorrBlock, 0, stream>>>(f, g, H, W, C, win, out);
        return cudaGetLastError();
    }
    const dim3 grid = xcorr_grid(H, W, C);
    const int rpc = (int)(((int64_t)H + grid.y - 1) / grid.y);
    xcorr_moments<<<grid, kXcorrBlock, 0, stream>>>(f, g, H, W, C, rpc, win, (double*)scratch);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    xcorr_windows<<<win.n, kXcorrBlock, 0, stream>>>((const double*)scratch, (int)(grid.x * grid.y), H, C, win, out);
    return cudaGetLastError();
}

// The columns inside a field of view are those about the image's centre whose
// angle is small enough, and the angle grows from the centre to either side:
// both ends are found by bisection (the search over all columns took an atan
// a column, some 20 us of host time for three fields of view of 512 columns).
void fov_windows(int W, double hfov_deg, const double* fov_deg, int n_fov, Windows* win)
{
    const double tx = tan(0.5 * hfov_deg * kPi / 180.0);
    const int mid = W / 2;                    // columns below it lie left of the centre
    win->n = n_fov;
    for (int q = 0; q < n_fov; ++q) {
        auto inside = [&](int j) {
            const double px = 2.0 * (j + 0.5) / W - 1.0;
            const double alpha = atan(fabs(px) * tx) * 180.0 / kPi;
            return alpha <= 0.5 * fov_deg[q] + 1e-9;
        };
        int a = 0, b = mid;                   // the first column inside in [0, mid], or mid
        while (a < b) {
            const int m = (a + b) / 2;
            if (inside(m)) b = m;
            else a = m + 1;
        }
        int c = mid - 1, d = W - 1;           // the last column inside in [mid - 1, W - 1], or mid - 1
        while (c < d) {
            const int m = c + (d - c + 1) / 2;                // (c + d may pass 2^31)
            if (inside(m)) c = m;
            else d = m - 1;
        }
        // a == mid: none on the left; c == mid - 1: none on the right
        win->j0[q] = a;
        win->j1[q] = c + 1;
        if (win->j1[q] <= win->j0[q]) win->j0[q] = win->j1[q] = 0;
    }
}

}  // namespace grt

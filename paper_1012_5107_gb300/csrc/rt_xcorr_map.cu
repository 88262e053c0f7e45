// rt_xcorr_map.cu -- the cross-correlation function C(di, dj) of Eq. 15 over
// pixel shifts, its peak and its mean over several reference pairs (Sec. 5).
//
// Pass 1 forms, over the field-of-view window of columns j0..j1-1, the means
// of Eq. 14 and the denominator sum (f - <f>)^2 of Eq. 15: a block per image
// row and pair sums it in three floats (rt_moments.cuh), then a block per pair
// and channel adds the rows in FP64.
// Pass 2 is a direct correlation in tiles: a block stages chunks of 8 image
// rows x 128 columns of f, of one pair and channel, and the window of g that
// its shifts (di, dj) need (zero outside the field-of-view window, where the
// finite photographs have no values) in shared memory, and each thread
// accumulates the products of its few shifts over a chunk with FP32 FMA (see
// xmap_tiles; choose_plan says how many).
// Pass 3 adds, per shift, pair, channel and column chunk, the row chunks'
// sums with compensated (Kahan) FP32 summation, whose error is of the order
// of one FP32 rounding of the result, below the rounding already in each
// chunk's sum (FP64 adds are 64 times slower on this GPU).  Pass 4 adds the
// column chunks in FP64, divides by the denominators, stacks the channels
// (sum of numerators over sum of denominators) and averages the maps of the
// pairs; pass 5 finds the peak of the stacked mean map and its shift.
//
// Measured: +-32 shifts of a 512 x 512 x 3 pair 320 -> 215 us.  The tiles, 261 us
// of it, computed 80 x 80 shifts for the 65 x 65 wanted, 25 a thread; now the
// threads' shifts divide those wanted and the tiles take 150 us (72 us at the
// FP32 peak).  +-31 x +-3 shifts of two 326 x 164 pairs 139 -> 58 us, +-40 of two
// 300 x 400 x 3 pairs 1,095 -> 312 us.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

#include "rt_internal.h"
#include "rt_moments.cuh"

namespace grt {

constexpr int kMapRows = 8;       // image rows per chunk
constexpr int kMapCols = 128;     // image columns per chunk
constexpr int kMapThreads = 160;  // threads per block of the tiles, at most
constexpr int kMapMaxShift = 64;
// Shared memory of any plan (the largest over all shifts and heights: 107,284
// bytes).  The limit of a kernel is the process's, so it is set to this once and
// not to a call's own size: a smaller call of another thread would lower it
// between a larger call's setting and its launch.
constexpr size_t kMapSmem = 108 * 1024;

// How a launch of the tiles is laid out: a thread owns RI x RJ shifts, gi x gj
// threads the shifts of a chunk, of which a block takes git along di; kc row
// chunks share a block and its window of g, gc floats a row.
struct MapPlan {
    int ri, rj, gi, gj, git, kc, gc, threads;
    size_t smem;
};
constexpr int kMapMaxPairs = 64;

struct MapImages {
    const float* f[kMapMaxPairs];
    const float* g[kMapMaxPairs];
};

constexpr int kMomRows = 1;       // image rows per block of pass 1
constexpr int kMomBlock = 256;

// A window row's values, (i W + j0) C ... (i W + j1) C, are contiguous, and
// the stride T is a multiple of C, so thread t meets only channel t mod C;
// the block's per-channel sums go to part[((pair nchunks + chunk) C + c) 3 + q]
// (q: sum f, sum g, sum f^2).
__global__ void __launch_bounds__(kMomBlock) xmap_moment_rows(MapImages im, int H, int W, int C, int j0, int j1,
                                                              int nchunks, double* __restrict__ part)
{
    __shared__ double red[3][kMomBlock];
    const int chunk = blockIdx.x, pair = blockIdx.y;
    const float* f = im.f[pair];
    const float* g = im.g[pair];
    const int T = (kMomBlock / C) * C;
    const int len = (j1 - j0) * C;
    const int t = threadIdx.x;
    const int i0 = chunk * kMomRows, i1 = min(H, i0 + kMomRows);
    Z3 s1 = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, s2 = s1;   // (f, g) and (f^2, -)
    int odd = 0;
    if (t < T) {
        for (int i = i0; i < i1; ++i) {
            const int64_t base = ((int64_t)i * W + j0) * C;
#pragma unroll 4
            for (int e = t; e < len; e += T) {
                const float a = __ldg(f + base + e), b = __ldg(g + base + e);
                odd |= !(xcorr_plain(a) && xcorr_plain(b));
                const F2 p = two_prod(a, a);
                xcorr_add(s1, float2{a, b});
                xcorr_add(s2, float2{p.h, 0.0f});
                xcorr_low(s2, float2{p.l, 0.0f});
            }
        }
    }
    double sf = join_x(s1), sg = join_y(s1), sff = join_x(s2);
    if (__syncthreads_or(odd)) {                                  // outside the three-float range: in FP64
        sf = sg = sff = 0.0;
        if (t < T)
            for (int i = i0; i < i1; ++i) {
                const int64_t base = ((int64_t)i * W + j0) * C;
                for (int e = t; e < len; e += T) {
                    const double a = __ldg(f + base + e), b = __ldg(g + base + e);
                    sf += a;
                    sg += b;
                    sff += a * a;
                }
            }
    }
    red[0][t] = sf;
    red[1][t] = sg;
    red[2][t] = sff;
    __syncthreads();
    // the threads of a channel in two rounds of additions
    constexpr int kWays = 16;
    double acc = 0.0;
    const int way = t % kWays, o = t / kWays, q = o / C, c = o - q * C;
    if (o < 3 * C)
        for (int k = c + way * C; k < T; k += kWays * C) acc += red[q][k];
    for (int d = kWays / 2; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d, kWays);
    if (o < 3 * C && way == 0) part[(((int64_t)pair * nchunks + chunk) * C + c) * 3 + q] = acc;
}
static_assert(16 * 3 * 4 <= kMomBlock, "sixteen threads per channel and sum");

// Block per (pair, channel): the chunks' sums, then the statistics.
__global__ void __launch_bounds__(128) xmap_moment_stats(const double* __restrict__ part, int H, int C, int j0,
                                                         int j1, int nchunks, double* __restrict__ stats)
{
    const int pc = blockIdx.x, pair = pc / C, c = pc % C;
    double v[3] = {0.0, 0.0, 0.0};
    for (int k = threadIdx.x; k < nchunks; k += blockDim.x) {
        const double* p = part + (((int64_t)pair * nchunks + k) * C + c) * 3;
        v[0] += p[0];
        v[1] += p[1];
        v[2] += p[2];
    }
    __shared__ double red[3][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int q = 0; q < 3; ++q) {
        double x = v[q];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) red[q][warp] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[3];
        for (int q = 0; q < 3; ++q) t[q] = red[q][0] + red[q][1] + red[q][2] + red[q][3];
        const double N = (double)H * (double)(j1 - j0);
        const double mf = t[0] / N, mg = t[1] / N;          // Eq. 14
        stats[3 * pc + 0] = mf;
        stats[3 * pc + 1] = mg;
        stats[3 * pc + 2] = t[2] - t[0] * mf;               // sum (f - <f>)^2, Eq. 15 denominator
    }
}

// A thread owns the shifts (di0 + a, dj0 + b), a < RI, b < RJ, of one chunk.
// The product f(i, j) g(i + di, j + dj) of chunk row r and column q reads
// g_s[r + a][q + b] of its window; along q each of the RI g rows slides by one
// column, held in registers by position modulo RJ, so a column costs one
// broadcast f load and RI g loads for RI RJ FMAs: shared memory delivers one
// load a cycle to the SM's four FMA pipes, which 5 x 5 shifts a thread all but
// used up.  The chunk's sum per shift is FP32 (8 x 128 products, in that
// order); part[((pc nchunks + chunk) nshift + s)], chunk = rc ncc + cc.
template <int RI, int RJ>
__global__ void __launch_bounds__(kMapThreads, 3) xmap_tiles(MapImages im, const double* __restrict__ stats, int H,
                                                             int W, int C, int j0, int j1, int max_di, int max_dj,
                                                             int nrc, int ncc, MapPlan pl, float* __restrict__ part)
{
    extern __shared__ float map_smem[];
    const int GC = pl.gc, rows_f = pl.kc * kMapRows, rows_g = rows_f + pl.git * RI - 1;
    float* g_s = map_smem;                                   // [rows_g][GC]
    float* f_s = map_smem + (size_t)rows_g * GC;             // [rows_f][kMapCols]
    const int ndi = 2 * max_di + 1, ndj = 2 * max_dj + 1;
    const int tiles = (pl.gi + pl.git - 1) / pl.git;
    const int tile = blockIdx.x % tiles, group = blockIdx.x / tiles;
    const int cc = group % ncc, rc0 = (group / ncc) * pl.kc;
    const int pc = blockIdx.y;
    const int pair = pc / C, c = pc % C;
    const float* f = im.f[pair];
    const float* g = im.g[pair];
    const float mf = (float)stats[3 * pc + 0], mg = (float)stats[3 * pc + 1];
    const int di_lo = -max_di + tile * pl.git * RI, dj_lo = -max_dj;
    const int i0 = rc0 * kMapRows, jc = j0 + cc * kMapCols;
    // rows by warps, eight loads in flight a lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    for (int r = warp; r < rows_f; r += nwarp) {
        const int i = i0 + r;
        float v[kMapCols / 32];
#pragma unroll
        for (int k = 0; k < kMapCols / 32; ++k) {
            const int j = jc + lane + 32 * k;
            v[k] = (i < H && j < j1) ? __ldg(f + ((int64_t)i * W + j) * C + c) - mf : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < kMapCols / 32; ++k) f_s[r * kMapCols + lane + 32 * k] = v[k];
    }
    for (int r = warp; r < rows_g; r += nwarp) {
        const int i = i0 + di_lo + r;
        const bool row = i >= 0 && i < H;
        const float* gi = g + (int64_t)i * W * C + c;
        for (int q0 = lane; q0 < GC; q0 += 256) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int j = jc + dj_lo + q0 + 32 * k;
                v[k] = (row && j >= j0 && j < j1) ? __ldg(gi + (int64_t)j * C) - mg : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (q0 + 32 * k < GC) g_s[r * GC + q0 + 32 * k] = v[k];
        }
    }
    __syncthreads();
    const int units = pl.git * pl.gj;
    const int kc = threadIdx.x / units, u = threadIdx.x - kc * units;
    const int ui = u / pl.gj, uj = u - ui * pl.gj;
    const int rc = rc0 + kc;
    if (kc >= pl.kc || rc >= nrc || tile * pl.git + ui >= pl.gi) return;
    float acc[RI][RJ];
#pragma unroll
    for (int a = 0; a < RI; ++a)
#pragma unroll
        for (int b = 0; b < RJ; ++b) acc[a][b] = 0.0f;
    for (int r = 0; r < kMapRows; ++r) {
        const float* fr = f_s + (kc * kMapRows + r) * kMapCols;
        const float* gr = g_s + (size_t)(kc * kMapRows + r + ui * RI) * GC + uj * RJ;
        float win[RI][RJ];
#pragma unroll
        for (int a = 0; a < RI; ++a)
#pragma unroll
            for (int b = 0; b < RJ; ++b) win[a][b] = gr[a * GC + b];
        // column q0 + v with the window's column b at position (v + b) mod RJ;
        // the f values of the next RJ columns are loaded ahead
        float fv[RJ];
#pragma unroll
        for (int v = 0; v < RJ; ++v) fv[v] = fr[v];
        auto column = [&](int q0, int v) {
            const float x = fv[v];
            fv[v] = fr[q0 + v + RJ];                              // (past the row at its end: not used)
#pragma unroll
            for (int a = 0; a < RI; ++a) {
#pragma unroll
                for (int b = 0; b < RJ; ++b) acc[a][b] = fmaf(x, win[a][(v + b) % RJ], acc[a][b]);
                win[a][v] = gr[a * GC + q0 + v + RJ];
            }
        };
#pragma unroll 1
        for (int q0 = 0; q0 + RJ <= kMapCols; q0 += RJ)
#pragma unroll
            for (int v = 0; v < RJ; ++v) column(q0, v);
#pragma unroll
        for (int v = 0; v < kMapCols % RJ; ++v) column(kMapCols - kMapCols % RJ, v);
    }
    const int64_t nshift = (int64_t)ndi * ndj, nchunks = (int64_t)nrc * ncc;
    float* o = part + ((int64_t)pc * nchunks + (int64_t)rc * ncc + cc) * nshift;
#pragma unroll
    for (int a = 0; a < RI; ++a) {
        const int di = di_lo + ui * RI + a;
#pragma unroll
        for (int b = 0; b < RJ; ++b) {
            const int dj = dj_lo + uj * RJ + b;
            if (di <= max_di && dj <= max_dj) o[(int64_t)(di + max_di) * ndj + (dj + max_dj)] = acc[a][b];
        }
    }
}

// Thread per (pair and channel pc, column chunk cc, shift s): the row chunks'
// sums, compensated; colsum[(pc ncc + cc) nshift + s] = sum - compensation.
__global__ void __launch_bounds__(256) xmap_sum(const float* __restrict__ part, int nrc, int ncc, int64_t n,
                                                int nshift, double* __restrict__ colsum)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int s = (int)(t % nshift);
    const int64_t pq = t / nshift;
    const int64_t pc = pq / ncc, cc = pq % ncc;
    const float* p = part + ((pc * nrc * ncc) + cc) * nshift + s;
    const int64_t stride = (int64_t)ncc * nshift;
    float sum = 0.0f, comp = 0.0f;
#pragma unroll 8
    for (int k = 0; k < nrc; ++k) {
        const float y = p[k * stride] - comp;
        const float u = sum + y;
        comp = (u - sum) - y;
        sum = u;
    }
    colsum[t] = (double)sum - (double)comp;
}

// (one warp a block: the divisions, FP64, spread over the SMs)
__global__ void __launch_bounds__(32) xmap_finish(const double* __restrict__ colsum,
                                                   const double* __restrict__ stats, int n_pairs, int C, int ncc,
                                                   int nshift, double* __restrict__ out)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nshift) return;
    double mean[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int p = 0; p < n_pairs; ++p) {
        double num_all = 0.0, den_all = 0.0;
        for (int c = 0; c < C; ++c) {
            const int pc = p * C + c;
            double num = 0.0;
            for (int q = 0; q < ncc; ++q) num += colsum[((int64_t)pc * ncc + q) * nshift + s];
            const double den = stats[3 * pc + 2];
            mean[c] += num / den;
            num_all += num;
            den_all += den;
        }
        mean[C] += num_all / den_all;
    }
    for (int c = 0; c <= C; ++c) out[(int64_t)s * (C + 1) + c] = mean[c] / (double)n_pairs;
}

// Peak of the stacked-channel map: largest value, the first in row-major
// order (di, then dj ascending) among equal ones.  Values are compared as
// integers of the same order (FP64 compares run on the FP64 pipe); NaN is
// below all.
__device__ __forceinline__ long long xmap_key(double v)
{
    const long long u = __double_as_longlong(v);
    const long long k = u >= 0 ? u : (long long)0x8000000000000000ull - u;      // -0.0 as 0.0
    return v == v ? k : (long long)0x8000000000000000ull;
}

__global__ void __launch_bounds__(1024) xmap_peak(const double* __restrict__ map, int C, int max_di, int max_dj,
                                                  double* __restrict__ peak)
{
    const int ndj = 2 * max_dj + 1, nshift = (2 * max_di + 1) * ndj;
    long long best = (long long)0x8000000000000000ull;
    int bi = nshift;
    for (int s = threadIdx.x; s < nshift; s += blockDim.x) {
        const long long v = xmap_key(map[(int64_t)s * (C + 1) + C]);
        if (v > best) { best = v; bi = s; }
    }
    __shared__ long long sv[32];
    __shared__ int si[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto reduce = [&]() {
        for (int o = 16; o > 0; o >>= 1) {
            const long long ov = __shfl_down_sync(0xffffffffu, best, o);
            const int oi = __shfl_down_sync(0xffffffffu, bi, o);
            if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
        }
    };
    reduce();
    if (lane == 0) { sv[warp] = best; si[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
        best = sv[lane];
        bi = si[lane];
        reduce();
        if (lane == 0) {
            peak[0] = bi < nshift ? map[(int64_t)bi * (C + 1) + C] : -INFINITY;
            peak[1] = (double)(bi / ndj - max_di);
            peak[2] = (double)(bi % ndj - max_dj);
        }
    }
}

// Layout of the tiles for ri x rj shifts a thread.
static MapPlan map_plan(int ri, int rj, int ndi, int ndj, int nrc)
{
    MapPlan p;
    p.ri = ri;
    p.rj = rj;
    p.gi = (ndi + ri - 1) / ri;
    p.gj = (ndj + rj - 1) / rj;
    const int tiles = (p.gi * p.gj + kMapThreads - 1) / kMapThreads;
    p.git = (p.gi + tiles - 1) / tiles;
    while (p.git * p.gj > kMapThreads) --p.git;
    p.kc = std::max(1, std::min(std::min(nrc, 8), kMapThreads / (p.git * p.gj)));
    // row length of the window: ri gc = 1 (mod 32) puts the lanes of different
    // di groups on banks one apart, between those of the dj groups (rj apart)
    p.gc = kMapCols + p.gj * rj + 1;
    while ((ri * p.gc) % 32 != 1) ++p.gc;
    auto bytes = [&] {
        return sizeof(float) * ((size_t)(p.kc * kMapRows + p.git * ri - 1) * p.gc + (size_t)p.kc * kMapRows * kMapCols + 16);
    };
    while (p.kc > 1 && bytes() > (size_t)74 * 1024) --p.kc;        // three blocks per SM
    p.smem = bytes();
    // few shifts keep few threads busy, but the block's window wants loading
    p.threads = std::max(128, (p.kc * p.git * p.gj + 31) / 32 * 32);
    return p;
}

// The shifts a thread owns: few enough that the launch fills the chip, many
// enough to load little.  The cost is the blocks of the fullest SM times a
// block's warps on its scheduler times the cycles of a column (FMAs and loads
// to issue, or the SM's shared memory delivering one load a cycle to four
// schedulers), and the block's loads.
static MapPlan choose_plan(int ndi, int ndj, int nrc, int ncc, int npc)
{
    constexpr int kSMs = 152;
    MapPlan best = {};
    double least = 1e300;
    for (int ri : {1, 3})
        for (int rj : {3, 5, 9, 13}) {
            const MapPlan p = map_plan(ri, rj, ndi, ndj, nrc);
            const int64_t blocks = (int64_t)((p.gi + p.git - 1) / p.git) * ((nrc + p.kc - 1) / p.kc) * ncc * npc;
            const int warps = (p.kc * p.git * p.gj + 31) / 32;
            const double column = std::max(warps / 4.0 * (ri * rj + ri + 1), (double)std::max(warps, 4) * (ri + 1));
            const double load = (double)p.smem / (4.0 * p.threads) * 60.0;
            const double cost = (double)((blocks + kSMs - 1) / kSMs) * (column * kMapRows * kMapCols + load);
            if (cost < least) { least = cost; best = p; }
        }
    return best;
}

template <int RI, int RJ>
static cudaError_t launch_tiles(cudaStream_t st, const MapPlan& p, const MapImages& im, const double* stats, int H,
                               int W, int C, int j0, int j1, int max_di, int max_dj, int nrc, int ncc, int npc,
                               float* part)
{
    if (p.ri != RI || p.rj != RJ) return cudaSuccess;
    if (p.smem > kMapSmem) return cudaErrorInvalidValue;
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done.load() & bit)) {
        e = cudaFuncSetAttribute(xmap_tiles<RI, RJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMapSmem);
        if (e != cudaSuccess) return e;
        done.fetch_or(bit);
    }
    const dim3 grid((unsigned)(((p.gi + p.git - 1) / p.git) * ((nrc + p.kc - 1) / p.kc) * ncc), npc);
    xmap_tiles<RI, RJ><<<grid, p.threads, p.smem, st>>>(im, stats, H, W, C, j0, j1, max_di, max_dj, nrc, ncc, p, part);
    return cudaGetLastError();
}

}  // namespace grt

using namespace grt;

extern "C" int rt_xcorr_map(const float* const* d_f, const float* const* d_g, int32_t n_pairs, int32_t height,
                            int32_t width, int32_t channels, double fov_deg, double hfov_deg, int32_t max_di,
                            int32_t max_dj, double* d_map, double* d_peak, void* stream)
{
    if (!d_f || !d_g || !d_map) { set_error("null pointer argument"); return RT_EINVAL; }
    if (n_pairs < 1 || n_pairs > kMapMaxPairs) { set_error("n_pairs must be 1..%d", kMapMaxPairs); return RT_EINVAL; }
    for (int p = 0; p < n_pairs; ++p)
        if (!d_f[p] || !d_g[p]) { set_error("image pointer of pair %d is NULL", p); return RT_EINVAL; }
    if (height < 1 || width < 1) { set_error("height and width must be >= 1"); return RT_EINVAL; }
    if (channels < 1 || channels > 4) { set_error("channels must be 1..4"); return RT_EINVAL; }
    if (max_di < 0 || max_di > kMapMaxShift || max_dj < 0 || max_dj > kMapMaxShift) {
        set_error("max_di and max_dj must be 0..%d", kMapMaxShift);
        return RT_EINVAL;
    }
    if (!(hfov_deg > 0.0 && hfov_deg < 180.0)) { set_error("hfov_deg must be in (0, 180)"); return RT_EINVAL; }
    if (!(fov_deg >= 0.0)) { set_error("fov_deg must be >= 0"); return RT_EINVAL; }
    Windows win;
    fov_windows(width, hfov_deg, &fov_deg, 1, &win);
    const int j0 = win.j0[0], j1 = win.j1[0];
    if (j1 <= j0) { set_error("the field of view holds no pixel column"); return RT_EINVAL; }
    MapImages im;
    for (int p = 0; p < n_pairs; ++p) { im.f[p] = d_f[p]; im.g[p] = d_g[p]; }
    const int ndi = 2 * max_di + 1, ndj = 2 * max_dj + 1, nshift = ndi * ndj;
    const int nrc = (height + kMapRows - 1) / kMapRows;
    const int ncc = (j1 - j0 + kMapCols - 1) / kMapCols;
    if ((int64_t)nrc * ncc > 65535) {
        set_error("rt_xcorr_map: %d x %d window chunks of %d x %d pixels exceed 65535", nrc, ncc, kMapRows, kMapCols);
        return RT_EINVAL;
    }
    const int nchunks = nrc * ncc;
    const int npc = n_pairs * channels;
    cudaStream_t st = (cudaStream_t)stream;
    const int mchunks = (height + kMomRows - 1) / kMomRows;
    double* stats = nullptr;
    double* partial = nullptr;
    // the moment sums of pass 1 (double) share the buffer of pass 2's chunk
    // sums (float), which they precede; the buffer holds the larger of the
    // two, then pass 3's column-chunk sums (double)
    const size_t chunk_bytes = (std::max(sizeof(float) * (size_t)npc * nchunks * nshift,
                                         sizeof(double) * (size_t)n_pairs * mchunks * channels * 3) + 255) &
                               ~(size_t)255;
    const size_t ncol = (size_t)npc * ncc * nshift;
    const size_t part_bytes = chunk_bytes + sizeof(double) * (ncol + 3 * (size_t)npc);
    cudaError_t e = scratch_alloc((void**)&partial, part_bytes, st);
    if (e == cudaSuccess) stats = (double*)((char*)partial + chunk_bytes) + ncol;
    if (e == cudaSuccess) {
        xmap_moment_rows<<<dim3(mchunks, n_pairs), kMomBlock, 0, st>>>(im, height, width, channels, j0, j1, mchunks,
                                                                        partial);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        xmap_moment_stats<<<npc, 128, 0, st>>>(partial, height, channels, j0, j1, mchunks, stats);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        const MapPlan p = choose_plan(ndi, ndj, nrc, ncc, npc);
        float* part = (float*)partial;
#define RT_TILES(RI, RJ)                                                                                              \
    if (e == cudaSuccess)                                                                                             \
        e = launch_tiles<RI, RJ>(st, p, im, stats, height, width, channels, j0, j1, max_di, max_dj, nrc, ncc, npc, part)
        RT_TILES(1, 3); RT_TILES(1, 5); RT_TILES(1, 9); RT_TILES(1, 13);
        RT_TILES(3, 3); RT_TILES(3, 5); RT_TILES(3, 9); RT_TILES(3, 13);
#undef RT_TILES
    }
    double* colsum = partial ? (double*)((char*)partial + chunk_bytes) : nullptr;
    if (e == cudaSuccess) {
        xmap_sum<<<(unsigned)((ncol + 255) / 256), 256, 0, st>>>((const float*)partial, nrc, ncc, (int64_t)ncol,
                                                                  nshift, colsum);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        xmap_finish<<<(nshift + 31) / 32, 32, 0, st>>>(colsum, stats, n_pairs, channels, ncc, nshift, d_map);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && d_peak) {
        xmap_peak<<<1, 1024, 0, st>>>(d_map, channels, max_di, max_dj, d_peak);
        e = cudaGetLastError();
    }
    if (partial) cudaFreeAsync(partial, st);
    if (e != cudaSuccess) {
        set_error("rt_xcorr_map: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? RT_ENOMEM : RT_ECUDA;
    }
    return RT_OK;
}

// k_windows.cu -- from the per-arm maps to the fine search windows (Sec. III-D, Eq. 11):
// sequential fusion with threshold phi, median hole filling (Jacobi passes), borders on
// the fine grid and the exclusive scan giving the padded row offsets.
//
// Up to two filling passes (the workloads') run in one kernel with the fusion and the windows, on
// tiles of 32 x 8 pixels with a halo of a pixel per pass, and the tile sums of the scan are added up
// there: seven launches of a few us each became two.  With the cost and path sums cleared beside the
// loads of the kernels before them, a 5x5 x 64^2 depth call takes 161 us instead of 185, the initial
// pass of 9x9 x 512^2 731 us instead of 762.  More passes would work on halos as large as the tile.
//
// D_init is kept in fixed point, in units of 1/8 coarse label: with at most four maps the
// running pairwise average m <- (m + 8 k_i) / 2 stays an exact integer (8k1, 4(k1+k2), ...),
// and -1 marks a discarded pixel.
#include "lfsgm_internal.cuh"

namespace lfsgm {
namespace {

__device__ __forceinline__ int fuse_pixel(const int *__restrict__ maps, int narms, int N, double phi8, int p) {
    int k[4];
#pragma unroll
    for (int i = 0; i < 4; i++) k[i] = i < narms ? __ldg(maps + (size_t)i * N + p) : 0;
    int m = 8 * k[0];
    bool ok = true;
#pragma unroll
    for (int i = 1; i < 4; i++)
        if (i < narms && ok) {
            const int mi = 8 * k[i];
            if ((double)abs(m - mi) < phi8) m = (m + mi) / 2;
            else ok = false;
        }
    return ok ? m : -1;
}

__global__ void fuse_kernel(const int *__restrict__ maps, int narms, int N, double phi, int *__restrict__ F) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) F[p] = fuse_pixel(maps, narms, N, 8.0 * phi, p);
}

// The lower middle of the valid (>= 0) values among the 8 neighbours of t (row stride ld), or -1.
__device__ __forceinline__ int fill_value(const int *t, int ld) {
    int vals[8], n = 0;
    for (int dy = -1; dy <= 1; dy++)
        for (int dx = -1; dx <= 1; dx++) {
            if (dx == 0 && dy == 0) continue;
            const int q = t[dy * ld + dx];
            if (q >= 0) {
                int j = n++;
                while (j > 0 && vals[j - 1] > q) { vals[j] = vals[j - 1]; j--; }
                vals[j] = q;
            }
        }
    return n > 0 ? vals[(n - 1) / 2] : -1;
}

// One Jacobi pass: a discarded pixel takes the median (lower middle) of the valid values
// among its 8 neighbours in the input map; without valid neighbours it stays discarded.
__global__ void fill_kernel(const int *__restrict__ Fin, int *__restrict__ Fout, int H, int W) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= H * W) return;
    const int v = Fin[p];
    if (v >= 0) { Fout[p] = v; return; }
    const int x = p % W, y = p / W;
    int vals[8];
    int n = 0;
    for (int dy = -1; dy <= 1; dy++)
        for (int dx = -1; dx <= 1; dx++) {
            if (dx == 0 && dy == 0) continue;
            const int xx = x + dx, yy = y + dy;
            if (xx < 0 || xx >= W || yy < 0 || yy >= H) continue;
            const int q = Fin[yy * W + xx];
            if (q >= 0) {
                int j = n++;
                while (j > 0 && vals[j - 1] > q) { vals[j] = vals[j - 1]; j--; }
                vals[j] = q;
            }
        }
    Fout[p] = n > 0 ? vals[(n - 1) / 2] : -1;
}

// Borders (Eq. 11): nearest fine label gc = round_half_up(m (G-1) / (8 (Lc-1))), window
// [gc - R, gc + R] saturated to [0, G-1]; a discarded pixel gets the whole range, and so does
// every pixel in the boundary-less mode (Sec. IV-E; F is not read).  Rfar > 0 makes the
// threshold depth-dependent (Sec. IV-F proposes a larger one for small disparities): linear from
// Rfar at gc = 0 to R at gc = G-1, R(gc) = R + floor((2 (Rfar - R)(G-1-gc) + G-1) / (2 (G-1))).
// Edge test of the border exclusion (Sec. III-D) on the edge-padded reference view (a padded read
// is the clamped read): the 3 x 3 Sobel sums, their squares and the comparison in FP32 with
// explicit rounding, in the order the oracle uses, so both take the same decision.
__device__ __forceinline__ bool sobel_edge(const float *I, int sx, int sy, float t) {
    const float q0 = I[-sy - sx], q1 = I[-sy], q2 = I[-sy + sx];
    const float q3 = I[-sx], q5 = I[sx];
    const float q6 = I[sy - sx], q7 = I[sy], q8 = I[sy + sx];
    const float gx = __fsub_rn(__fadd_rn(__fadd_rn(q2, __fmul_rn(2.0f, q5)), q8),
                               __fadd_rn(__fadd_rn(q0, __fmul_rn(2.0f, q3)), q6));
    const float gy = __fsub_rn(__fadd_rn(__fadd_rn(q6, __fmul_rn(2.0f, q7)), q8),
                               __fadd_rn(__fadd_rn(q0, __fmul_rn(2.0f, q1)), q2));
    return __fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)) > __fmul_rn(t, t);
}

// What the windows depend on besides D_init.
struct WindowArgs {
    int G, Lc, R, Rfar;
    const float *ref_pad;             // the padded reference view (channels interleaved), for the edge test
    int C, P, Wp;
    float edge_t;
    int *lo, *cnt;
    float *dinit;                     // nullable
    unsigned long long *tsum;         // padded counts per 1024 pixels, zeroed before
};

// The window of pixel p with D_init v (-1: discarded); returns its padded count.
__device__ __forceinline__ int window_of(const WindowArgs &a, int p, int x, int y, int v) {
    // an edge in any channel of the padded reference view (colour: one float4 per pixel, the
    // channels interleaved)
    bool edge = false;
    if (a.edge_t > 0.f) {
        const int sx = a.C == 1 ? 1 : 4;
        const float *q = a.ref_pad + ((size_t)(y + a.P) * a.Wp + (x + a.P)) * sx;
        for (int ch = 0; ch < a.C && !edge; ch++) edge = sobel_edge(q + ch, sx, sx * a.Wp, a.edge_t);
    }
    const int G = a.G;
    int l, n;
    if (v < 0 || edge) {
        l = 0;
        n = G;
        if (a.dinit) a.dinit[p] = v < 0 ? __int_as_float(0x7fc00000) : 0.125f * (float)v;
    } else {
        const long long num = (long long)v * (G - 1);
        const long long den = 8LL * (a.Lc - 1);
        const long long gc = (2 * num + den) / (2 * den);
        long long r = a.R;
        if (a.Rfar > 0) {
            const long long dg = G - 1, t = 2 * (long long)(a.Rfar - a.R) * (dg - gc) + dg;
            long long q = t / (2 * dg);
            if (t % (2 * dg) != 0 && t < 0) q--;          // floor division
            r = a.R + q;
        }
        long long lo_ = gc - r, hi_ = gc + r;
        if (lo_ < 0) lo_ = 0;
        if (hi_ > G - 1) hi_ = G - 1;
        l = (int)lo_;
        n = (int)(hi_ - lo_ + 1);
        if (a.dinit) a.dinit[p] = 0.125f * (float)v;
    }
    a.lo[p] = l;
    a.cnt[p] = n;
    return (n + 3) & ~3;
}

constexpr int kScanTile = 1024;

// Adds the padded counts of a warp's pixels (p >= 0) to their scan tiles.
__device__ __forceinline__ void add_tile_sums(unsigned long long *tsum, int p, int pad) {
    const int tile = p >= 0 ? p / kScanTile : -1;
    const int first = __reduce_max_sync(0xffffffffu, tile);
    if (__all_sync(0xffffffffu, tile < 0 || tile == first)) {
        const int sum = __reduce_add_sync(0xffffffffu, p >= 0 ? pad : 0);
        if ((threadIdx.x & 31) == 0 && first >= 0) atomicAdd(tsum + first, (unsigned long long)sum);
    } else if (p >= 0) {
        atomicAdd(tsum + tile, (unsigned long long)pad);
    }
}

__global__ void __launch_bounds__(256) windows_kernel(const int *__restrict__ F, int N, int W, WindowArgs a) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    int pad = 0;
    if (p < N) pad = window_of(a, p, p % W, p / W, F[p]);
    add_tile_sums(a.tsum, p < N ? p : -1, pad);
}

// Boundary-less: the windows are the whole range, the offsets multiples of its padded length.
__global__ void __launch_bounds__(256) whole_windows_kernel(int N, int G, int *__restrict__ lo, int *__restrict__ cnt,
                                                            long long *__restrict__ off, float *__restrict__ dinit) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > N) return;
    off[p] = (long long)p * ((G + 3) & ~3);
    if (p == N) return;
    lo[p] = 0;
    cnt[p] = G;
    if (dinit) dinit[p] = __int_as_float(0x7fc00000);
}

// Fusion, `passes` (0 .. 2) filling passes and the windows of a 32 x 8 tile; out of the image: -1, as
// a discarded pixel contributes nothing to a median.
__global__ void __launch_bounds__(256) fused_windows_kernel(const int *__restrict__ maps, int narms, int H, int W,
                                                            double phi, int passes, WindowArgs a) {
    constexpr int TW = 36, TH = 12;
    __shared__ int t[2][TH][TW];
    const int bx = (W + 31) >> 5, by = blockIdx.x / bx;                      // (one grid dimension: images of any height)
    const int xt = (blockIdx.x - by * bx) * 32, yt = by * 8;                 // the tile
    const int x0 = xt - passes, y0 = yt - passes;                            // image position of entry (0, 0)
    const int tid = threadIdx.y * 32 + threadIdx.x;
    for (int i = tid; i < TW * TH; i += 256) {
        const int ty = i / TW, tx = i - ty * TW, x = x0 + tx, y = y0 + ty;
        const bool in = tx < 32 + 2 * passes && ty < 8 + 2 * passes && x >= 0 && x < W && y >= 0 && y < H;
        t[0][ty][tx] = in ? fuse_pixel(maps, narms, H * W, 8.0 * phi, y * W + x) : -1;
    }
    __syncthreads();
    for (int k = 0; k < passes; k++) {
        const int w = 32 + 2 * (passes - 1 - k), h = 8 + 2 * (passes - 1 - k);   // from entry (k + 1, k + 1) on
        for (int i = tid; i < w * h; i += 256) {
            const int ty = i / w + k + 1, tx = i % w + k + 1, x = x0 + tx, y = y0 + ty;
            int v = t[k & 1][ty][tx];
            if (v < 0 && x >= 0 && x < W && y >= 0 && y < H) v = fill_value(&t[k & 1][ty][tx], TW);
            t[(k + 1) & 1][ty][tx] = v;
        }
        __syncthreads();
    }
    const int x = xt + threadIdx.x, y = yt + threadIdx.y;
    const bool in = x < W && y < H;
    int pad = 0;
    if (in) pad = window_of(a, y * W + x, x, y, t[passes & 1][threadIdx.y + passes][threadIdx.x + passes]);
    add_tile_sums(a.tsum, in ? y * W + x : -1, pad);
}

// Exclusive scan of the padded counts over tiles of 1024 entries, whose sums the windows kernels have
// added up: per tile a scan plus the sum of the tiles before it (images of many tiles: of a scan of
// the tile sums by one CTA).
constexpr int kTopTiles = kScanTile;   // one sum per thread

__device__ __forceinline__ long long block_exclusive_scan(long long v, long long *wsum, long long *total) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    long long inc = v;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        long long w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    const long long ex = inc - v + (wid > 0 ? wsum[wid - 1] : 0);
    if (total) *total = wsum[(blockDim.x >> 5) - 1];
    __syncthreads();
    return ex;
}

__global__ void __launch_bounds__(kScanTile) scan_tile_offsets(long long *__restrict__ tsum, int ntiles) {
    __shared__ long long wsum[32];
    long long carry = 0;
    for (int base = 0; base < ntiles; base += kScanTile) {
        const int i = base + threadIdx.x;
        const long long v = i < ntiles ? tsum[i] : 0;
        long long total;
        const long long ex = block_exclusive_scan(v, wsum, &total);
        if (i < ntiles) tsum[i] = carry + ex;
        carry += total;
    }
}

__global__ void __launch_bounds__(kScanTile) scan_apply(const int *__restrict__ cnt, int N, const long long *__restrict__ tsum,
                                                        bool scanned, long long *__restrict__ off) {
    __shared__ long long wsum[32];
    const int i = blockIdx.x * kScanTile + threadIdx.x;
    const long long v = i < N ? (__ldg(cnt + i) + 3) & ~3 : 0;
    long long before = 0;
    if (scanned) {
        before = __ldg(tsum + blockIdx.x);
    } else {
        // the tiles before this one
        long long s = 0, total;
        for (int t = threadIdx.x; t < (int)blockIdx.x; t += kScanTile) s += __ldg(tsum + t);
        block_exclusive_scan(s, wsum, &total);
        before = total;
    }
    const long long ex = block_exclusive_scan(v, wsum, nullptr);
    const long long o = before + ex;
    if (i < N) off[i] = o;
    if (i == N - 1) off[N] = o + v;
}

}  // namespace

cudaError_t launch_fuse(cudaStream_t s, const int *maps, int narms, int N, double phi, int *F) {
    fuse_kernel<<<(N + 255) / 256, 256, 0, s>>>(maps, narms, N, phi, F);
    return cudaGetLastError();
}
cudaError_t launch_fill(cudaStream_t s, const int *Fin, int *Fout, int H, int W) {
    fill_kernel<<<(H * W + 255) / 256, 256, 0, s>>>(Fin, Fout, H, W);
    return cudaGetLastError();
}
static WindowArgs window_args(const WindowSetup &u) {
    WindowArgs a;
    a.G = u.G; a.Lc = u.Lc; a.R = u.R; a.Rfar = u.Rfar;
    a.ref_pad = u.ref_pad; a.C = u.C; a.P = u.P; a.Wp = u.Wp; a.edge_t = u.edge_t;
    a.lo = u.lo; a.cnt = u.cnt; a.dinit = u.dinit; a.tsum = (unsigned long long *)u.tsum;
    return a;
}
cudaError_t launch_whole_windows(cudaStream_t s, int N, int G, int *lo, int *cnt, long long *off, float *dinit) {
    whole_windows_kernel<<<N / 256 + 1, 256, 0, s>>>(N, G, lo, cnt, off, dinit);
    return cudaGetLastError();
}
cudaError_t launch_windows(cudaStream_t s, const int *F, int N, int W, const WindowSetup &u) {
    windows_kernel<<<(N + 255) / 256, 256, 0, s>>>(F, N, W, window_args(u));
    return cudaGetLastError();
}
cudaError_t launch_fused_windows(cudaStream_t s, const int *maps, int narms, int H, int W, double phi, int passes,
                                 const WindowSetup &u) {
    fused_windows_kernel<<<(W + 31) / 32 * ((H + 7) / 8), dim3(32, 8), 0, s>>>(maps, narms, H, W, phi, passes,
                                                                              window_args(u));
    return cudaGetLastError();
}
int scan_tiles(int N) { return (N + kScanTile - 1) / kScanTile; }
bool scan_needs_top(int N) { return scan_tiles(N) > kTopTiles; }

cudaError_t launch_scan_top(cudaStream_t s, long long *tsum, int N) {
    scan_tile_offsets<<<1, kScanTile, 0, s>>>(tsum, scan_tiles(N));
    return cudaGetLastError();
}
cudaError_t launch_scan_apply(cudaStream_t s, const int *cnt, int N, const long long *tsum, long long *off) {
    scan_apply<<<scan_tiles(N), kScanTile, 0, s>>>(cnt, N, tsum, scan_needs_top(N), off);
    return cudaGetLastError();
}

}  // namespace lfsgm

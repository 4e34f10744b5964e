// k_fine_cost.cu -- bounded fine cost volume (Sec. III-E, Eq. 12 with the census term of
// Eq. 15):
//   C(p,g) = w_l2 * sum_views |I_ref(p) - bilinear(I_uv, p + (u-uc, v-vc) d_g)|
//          + w_c  * sum_views HD(census_ref(p), census_uv(p + nearest shift)),
// over every view but the reference, for the labels g of p's window only.
//
// Generic form: one warp per pixel, lane j owns window slot j (label lo + j; wide windows
// loop in chunks of 32), and walks the views in the order v-major, u-minor.  The shift
// split of every (view, label) comes from the host-built FineTap table; taps and census
// words are read through the read-only cache.  Output rows are written coalesced,
// padding slots with 0.
#include "lfsgm_internal.cuh"

#include <algorithm>

namespace lfsgm {
namespace {

__global__ void __launch_bounds__(256) fine_cost_generic(const float *__restrict__ views,
                                                         const uint64_t *__restrict__ cen,
                                                         const FineTap *__restrict__ tab, int G,
                                                         int nviews, int H, int W, int ref,
                                                         const int *__restrict__ lo,
                                                         const int *__restrict__ cnt,
                                                         const long long *__restrict__ off, float wl2,
                                                         float wc, float *__restrict__ cost,
                                                         int *__restrict__ status) {
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const size_t N = (size_t)H * W;
    for (int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < (int)N; p += warps) {
        const int x = p % W, y = p / W;
        const int l0 = __ldg(lo + p), n = __ldg(cnt + p);
        const long long o = __ldg(off + p), row = __ldg(off + p + 1) - o;
        if (!window_ok(l0, n, G, row, status)) continue;
        const float Iref = __ldg(views + (size_t)ref * N + p);
        const uint64_t cr = __ldg(cen + (size_t)ref * N + p);
        const int npad = (int)min((long long)((n + 3) & ~3), row);
        for (int j = lane; j < npad; j += 32) {
            float acc = 0.f;
            if (j < n) {
                const int g = l0 + j;
                float sl2 = 0.f;
                int sc = 0;
                for (int view = 0; view < nviews; view++) {
                    if (view == ref) continue;
                    const FineTap t = load_tap(tab + (size_t)view * G + g);
                    const float *I = views + (size_t)view * N;
                    const int x0 = min(max(x + t.ox, 0), W - 1), x1 = min(max(x + t.ox + 1, 0), W - 1);
                    const int y0 = min(max(y + t.oy, 0), H - 1), y1 = min(max(y + t.oy + 1, 0), H - 1);
                    const float i00 = __ldg(I + (size_t)y0 * W + x0), i10 = __ldg(I + (size_t)y0 * W + x1);
                    const float i01 = __ldg(I + (size_t)y1 * W + x0), i11 = __ldg(I + (size_t)y1 * W + x1);
                    const float top = (1.f - t.fx) * i00 + t.fx * i10;
                    const float bot = (1.f - t.fx) * i01 + t.fx * i11;
                    const float smp = (1.f - t.fy) * top + t.fy * bot;
                    sl2 += fabsf(Iref - smp);
                    const int xn = min(max(x + t.nx, 0), W - 1), yn = min(max(y + t.ny, 0), H - 1);
                    sc += __popcll(cr ^ __ldg(cen + (size_t)view * N + (size_t)yn * W + xn));
                }
                acc = wl2 * sl2 + wc * (float)sc;
            }
            cost[o + j] = acc;
        }
    }
}

// The per-pixel form over a list of (pixel, chunk) items (the windows that the ranges of
// k_fine_rows.cu leave):
// one warp per item, lane = label of the chunk, taps read from the padded views and census words
// (no clamping needed) at linear offsets (oy Wp + ox, ny Wp + nx).  Each lane reads its label's
// table entry of a view with one coalesced 16-byte load (the warp's 32 entries are contiguous);
// two views per unrolled step keep their loads in flight together.  Colour (C > 1): the padded
// views hold one float4 per pixel (channels interleaved), so a bilinear tap of all channels is
// four 16-byte loads, and the census words are planes view * C + c; the l2 term is the Euclidean
// norm of the colour difference and the census term sums the channels' Hamming distances
// (Sec. III-B/C).
constexpr int kListWarps = 4;

// LEAN (grey): 32 registers for 16 CTAs of 128 threads per SM (a few spilled bytes); the grey
// list is latency-bound, and the extra warps took the bench light field's list from 0.241 to
// 0.193 ms, while the all-wide Middlebury-shaped list runs best with 40 registers and 12 CTAs
// (0.697 vs 0.722 ms): the speed knob picks.  Colour: 12 CTAs per SM (0.42 -> 0.37 ms against 9).
template <int C, bool LEAN>
__global__ void __launch_bounds__(32 * kListWarps, C == 3 ? 12 : (LEAN ? 16 : 12)) fine_cost_list(const float *__restrict__ views_pad,
                                                      const uint64_t *__restrict__ cen_pad, int P, int Wp, int Hp,
                                                      const int4 *__restrict__ ltab, int G, int nviews,
                                                      int W, int ref, const int *__restrict__ lo,
                                                      const int *__restrict__ cnt,
                                                      const long long *__restrict__ off, float wl2, float wc,
                                                      float *__restrict__ cost, const int2 *__restrict__ list,
                                                      const int *__restrict__ count,
                                                      const int *__restrict__ large) {
    if (large && __ldg(large) == 0) return;              // census_list has done the list
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const size_t HWp = (size_t)Hp * Wp;
    const int total = *count;
    const int nv1 = nviews - 1;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < total; t += warps) {
        const int2 item = list[t];
        const int p = item.x, chunk = item.y;
        const int l0 = __ldg(lo + p), n = __ldg(cnt + p);
        const long long o = __ldg(off + p), row = __ldg(off + p + 1) - o;
        if (!window_ok(l0, n, G, row, nullptr)) continue;      // items are pushed for valid windows only
        const int npad = (int)min((long long)((n + 3) & ~3), row);
        const int j = chunk * 32 + lane;
        const int x = p % W, y = p / W;
        const size_t base = (size_t)(y + P) * Wp + (x + P);
        float sl2 = 0.f;
        int sc = 0;
        if (j < n) {
            uint64_t cr[C];
#pragma unroll
            for (int ch = 0; ch < C; ch++) cr[ch] = __ldg(cen_pad + ((size_t)ref * C + ch) * HWp + base);
            const int4 *tg = ltab + l0 + j;
            if constexpr (C == 1) {
                const float Iref = __ldg(views_pad + (size_t)ref * HWp + base);
#pragma unroll 2
                for (int vi = 0; vi < nv1; vi++) {
                    const int view = vi + (vi >= ref);
                    const int4 tw = __ldg(tg + (size_t)view * G);     // linear tap offsets (x + Wp y), fx, fy
                    const size_t vb = (size_t)view * HWp + base;
                    const float tfx = __int_as_float(tw.z), tfy = __int_as_float(tw.w);
                    const float *q = views_pad + vb + tw.x;
                    const float i00 = __ldg(q), i10 = __ldg(q + 1), i01 = __ldg(q + Wp), i11 = __ldg(q + Wp + 1);
                    const float top = (1.f - tfx) * i00 + tfx * i10;
                    const float bot = (1.f - tfx) * i01 + tfx * i11;
                    sl2 += fabsf(Iref - ((1.f - tfy) * top + tfy * bot));
                    sc += __popcll(cr[0] ^ __ldg(cen_pad + vb + tw.y));
                }
            } else {
                const float4 *v4 = reinterpret_cast<const float4 *>(views_pad);
                const float4 Iref = __ldg(v4 + (size_t)ref * HWp + base);
#pragma unroll 2
                for (int vi = 0; vi < nv1; vi++) {
                    const int view = vi + (vi >= ref);
                    const int4 tw = __ldg(tg + (size_t)view * G);
                    const size_t pb = (size_t)view * HWp + base;
                    const float tfx = __int_as_float(tw.z), tfy = __int_as_float(tw.w);
                    const float4 *q = v4 + pb + tw.x;
                    const float4 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + Wp), d = __ldg(q + Wp + 1);
                    auto sample = [&](float i00, float i10, float i01, float i11) {
                        const float top = (1.f - tfx) * i00 + tfx * i10;
                        const float bot = (1.f - tfx) * i01 + tfx * i11;
                        return (1.f - tfy) * top + tfy * bot;
                    };
                    const float d0 = Iref.x - sample(a.x, b.x, c.x, d.x);
                    const float d1 = Iref.y - sample(a.y, b.y, c.y, d.y);
                    const float d2 = Iref.z - sample(a.z, b.z, c.z, d.z);
                    sl2 += sqrtf(fmaf(d2, d2, fmaf(d1, d1, d0 * d0)));
#pragma unroll
                    for (int ch = 0; ch < C; ch++)
                        sc += __popcll(cr[ch] ^ __ldg(cen_pad + ((size_t)view * C + ch) * HWp + base + tw.y));
                }
            }
        }
        if (j < npad) cost[o + j] = (j < n) ? wl2 * sl2 + wc * (float)sc : 0.f;
    }
}


// The cost without the l2 term (w_l2 = 0, the paper's census-only cost of real scenes; grey), while the
// views are small enough that 0 x l2 is 0 (`large` is not set: with a NaN or an infinity among the
// samples 0 x l2 is NaN, so the full list runs then).  7x1 x 555x650, 121 labels, every window the whole
// range: 722 us in the full list; 495 us in census_list alone (a few views an item: its loads' latency);
// most of it in census_runs.
//
// Runs of 32 pixels of a row whose windows are all the whole range (marked by row_tasks_kernel): one
// warp per run, lane = pixel.  A label's shift is the same for every pixel and changes only every few
// labels, so a view's Hamming distance is a step function of the label (as in the coarse cost): a word
// read, coalesced over the pixels, and a popcount only at the steps, added to a difference column in
// shared memory (two labels a word), prefix-summed, and the rows written through a 32 x 32 tile.
constexpr int kRunLabels = 96, kRunWarps = 4;
__global__ void __launch_bounds__(32 * kRunWarps) census_runs(const uint64_t *__restrict__ cen_pad, int P, int Wp,
                                                              int Hp, const int *__restrict__ ctab, int G, int nviews,
                                                              int H, int W, int ref,
                                                              const unsigned char *__restrict__ marks,
                                                              const long long *__restrict__ off, float wc,
                                                              float *__restrict__ cost) {
    __shared__ int cdiff[kRunWarps][kRunLabels / 2][32];
    __shared__ float tile[kRunWarps][32][33];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int bx = (W + 31) >> 5;
    const int run = blockIdx.x * kRunWarps + w;              // row-major over (row, run of the row)
    if (run >= bx * H || !__ldg(marks + run)) return;
    const int y = run / bx, x0 = (run - y * bx) << 5, x = min(x0 + lane, W - 1);
    const size_t HWp = (size_t)Hp * Wp, base = (size_t)(y + P) * Wp + (x + P);
    const int npx = min(32, W - x0);
    const long long o = __ldg(off + (size_t)y * W + x);
    const int npad = (int)min((long long)((G + 3) & ~3), __ldg(off + (size_t)y * W + x + 1) - o);
    const uint64_t cr = __ldg(cen_pad + (size_t)ref * HWp + base);
    int *cd = &cdiff[w][0][lane];
    for (int g0 = 0; g0 < G; g0 += kRunLabels) {
        const int ng = min(kRunLabels, G - g0);
#pragma unroll 4
        for (int i = 0; i < kRunLabels / 2; i++) cd[32 * i] = 0;
        for (int v = 0; v < nviews; v++) {
            if (v == ref) continue;
            const uint64_t *q = cen_pad + (size_t)v * HWp + base;
            const int *ot = ctab + (size_t)v * G + g0;
            int hp = 0, oprev = 0;
            for (int k0 = 0; k0 < ng; k0 += 32) {
                const int k = k0 + lane;
                const int ov = k < ng ? __ldg(ot + k) : 0;
                const int up = __shfl_up_sync(0xffffffffu, ov, 1);
                const int before = lane == 0 ? oprev : up;
                unsigned steps = __ballot_sync(0xffffffffu, k < ng && (k == 0 || ov != before));
                oprev = __shfl_sync(0xffffffffu, ov, 31);
                // the steps four at a time: their word loads are issued together
                while (steps) {
                    int bs[4];
                    uint64_t wv[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        bs[u] = steps ? __ffs(steps) - 1 : -1;          // warp-uniform
                        steps &= steps - 1;
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int so = __shfl_sync(0xffffffffu, ov, bs[u] & 31);
                        wv[u] = bs[u] >= 0 ? __ldg(q + so) : 0ull;
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        if (bs[u] < 0) break;
                        const int h = __popcll(cr ^ wv[u]);
                        const int kb = k0 + bs[u];
                        cd[32 * (kb >> 1)] += (int)((unsigned)(h - hp) << (16 * (kb & 1)));
                        hp = h;
                    }
                }
            }
        }
        int sum = 0;
        for (int k0 = 0; k0 < ng; k0 += 32) {
#pragma unroll 4
            for (int k = 0; k < 32; k += 2) {
                // the word holds d(k) + d(k+1) 2^16 (two's complement, |d| < 2^15): split it exactly
                const int wd = cd[32 * ((k0 + k) >> 1)];
                const int d0 = (int)(short)(wd & 0xffff);
                sum += d0;
                tile[w][lane][k] = wc * (float)sum;
                sum += (wd - d0) >> 16;
                tile[w][lane][k + 1] = wc * (float)sum;
            }
            __syncwarp();
            const int j = g0 + k0 + lane;
#pragma unroll 4
            for (int q = 0; q < npx; q++) {
                const long long oq = __shfl_sync(0xffffffffu, o, q);
                const int nq = __shfl_sync(0xffffffffu, npad, q);
                if (j < nq) cost[oq + j] = j < G ? tile[w][q][lane] : 0.f;
            }
            __syncwarp();
        }
    }
}

// The other items: one warp per (pixel, 32-label chunk); per view a lane reads its label's offset
// (ctab: ny Wp + nx) and one census word.
__global__ void __launch_bounds__(32 * kListWarps) census_list(const uint64_t *__restrict__ cen_pad, int P, int Wp,
                                                               int Hp, const int *__restrict__ ctab, int G, int nviews,
                                                               int W, int ref, const int *__restrict__ lo,
                                                               const int *__restrict__ cnt,
                                                               const long long *__restrict__ off, float wc,
                                                               float *__restrict__ cost, const int2 *__restrict__ list,
                                                               const int *__restrict__ count,
                                                               const int *__restrict__ large) {
    if (__ldg(large)) return;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const size_t HWp = (size_t)Hp * Wp;
    const int total = *count;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < total; t += warps) {
        const int2 item = __ldg(list + t);
        const int p = item.x, chunk = item.y;
        const int l0 = __ldg(lo + p), n = __ldg(cnt + p);
        const long long o = __ldg(off + p), row = __ldg(off + p + 1) - o;
        if (!window_ok(l0, n, G, row, nullptr)) continue;      // items are pushed for valid windows only
        const int npad = (int)min((long long)((n + 3) & ~3), row);
        const int j = chunk * 32 + lane;
        const int x = p % W, y = p / W;
        const size_t base = (size_t)(y + P) * Wp + (x + P);
        int sc = 0;
        if (j < n) {
            const uint64_t cr = __ldg(cen_pad + (size_t)ref * HWp + base);
            const int *tg = ctab + l0 + j;
            const uint64_t *q = cen_pad + base;
            auto view = [&](int v) { return __popcll(cr ^ __ldg(q + (size_t)v * HWp + __ldg(tg + (size_t)v * G))); };
            int v = 0;
            // (the reference view's own distance, at shift 0, is 0)
            for (; v + 4 <= nviews; v += 4) sc += view(v) + view(v + 1) + view(v + 2) + view(v + 3);
            for (; v < nviews; v++) sc += view(v);
        }
        if (j < npad) cost[o + j] = j < n ? wc * (float)sc : 0.f;
    }
}

__global__ void list_all_kernel(const int *__restrict__ lo, const int *__restrict__ cnt,
                                const long long *__restrict__ off, int G, int2 *list, int *count, int N,
                                int *status, int min_cnt) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N && cnt[p] > min_cnt && window_ok(lo[p], cnt[p], G, off[p + 1] - off[p], status))
        push_chunks(list, count, p, cnt[p]);
}

}  // namespace

cudaError_t launch_list_all(cudaStream_t s, const int *lo, const int *cnt, const long long *off, int G, int2 *list,
                            int *count, int N, int *status, int min_cnt) {
    list_all_kernel<<<(N + 255) / 256, 256, 0, s>>>(lo, cnt, off, G, list, count, N, status, min_cnt);
    return cudaGetLastError();
}

cudaError_t launch_fine_cost_list(cudaStream_t s, const float *views_pad, const uint64_t *cen_pad, int P, int Wp,
                                  int Hp, const int4 *ltab, int G, int nviews, int C, int W, int ref,
                                  const int *lo, const int *cnt, const long long *off, float wl2, float wc,
                                  float *cost, const int2 *list, const int *count, int ctas_per_sm,
                                  const int *large) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // grid-stride over the items, by default with exactly the CTAs that are resident at once: the
    // warps then sweep the list (pixel order) once, together, and the views around the rows in
    // flight stay in L2; a second wave would sweep the whole image again (colour: 9 resident CTAs
    // per SM, 4.35 ms, against 4.92 ms with 24 and 6.48 ms with 12)
    // grey: the lean instantiation by default and for 16 or more CTAs per SM, the other one below
    const bool lean = C == 1 && (ctas_per_sm <= 0 || ctas_per_sm >= 16);
    auto kern = C == 3 ? fine_cost_list<3, false> : (lean ? fine_cost_list<1, true> : fine_cost_list<1, false>);
    int k = ctas_per_sm;
    if (k <= 0) {
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, kern, 32 * kListWarps, 0);
        if (e != cudaSuccess) return e;
        k = max(k, 1);
    }
    kern<<<sms * k, 32 * kListWarps, 0, s>>>(views_pad, cen_pad, P, Wp, Hp, ltab, G, nviews, W, ref, lo, cnt, off, wl2,
                                             wc, cost, list, count, large);
    return cudaGetLastError();
}

cudaError_t launch_census_runs(cudaStream_t s, const uint64_t *cen_pad, int P, int Wp, int Hp, const int *ctab, int G,
                               int nviews, int H, int W, int ref, const unsigned char *marks, const long long *off,
                               float wc, float *cost) {
    const long long runs = (long long)((W + 31) / 32) * H;
    census_runs<<<(unsigned)((runs + kRunWarps - 1) / kRunWarps), 32 * kRunWarps, 0, s>>>(
        cen_pad, P, Wp, Hp, ctab, G, nviews, H, W, ref, marks, off, wc, cost);
    return cudaGetLastError();
}

cudaError_t launch_census_list(cudaStream_t s, const uint64_t *cen_pad, int P, int Wp, int Hp, const int *ctab, int G,
                               int nviews, int W, int ref, const int *lo, const int *cnt, const long long *off, float wc,
                               float *cost, const int2 *list, const int *count, const int *large) {
    int dev = 0, sms = 0, k = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, census_list, 32 * kListWarps, 0);
    if (e != cudaSuccess) return e;
    census_list<<<sms * max(k, 1), 32 * kListWarps, 0, s>>>(cen_pad, P, Wp, Hp, ctab, G, nviews, W, ref, lo, cnt, off, wc,
                                                            cost, list, count, large);
    return cudaGetLastError();
}

cudaError_t launch_fine_cost(cudaStream_t s, const float *views, const uint64_t *cen, const FineTap *tab,
                             int G, int nviews, int H, int W, int ref, const int *lo, const int *cnt,
                             const long long *off, float wl2, float wc, float *cost, int *status) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int block = 256;
    const long long want = ((long long)H * W * 32 + block - 1) / block;
    const int grid = (int)(want < (long long)sms * 8 ? want : (long long)sms * 8);
    fine_cost_generic<<<grid, block, 0, s>>>(views, cen, tab, G, nviews, H, W, ref, lo, cnt, off, wl2,
                                             wc, cost, status);
    return cudaGetLastError();
}

}  // namespace lfsgm

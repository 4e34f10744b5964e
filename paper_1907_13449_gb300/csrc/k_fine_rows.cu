// k_fine_rows.cu -- block form of the bounded fine cost volume (Sec. III-E, Eq. 12 with the census
// term of Eq. 15) for the regular (narrow) windows; k_fine_cost.cu's list kernel takes the others.
//
// For a fixed view and fine label the shift (u-uc, v-vc) d_g is the same for every pixel, so the
// pixels of a run sweep one label range with a label index that is the same for all of them.
// row_tasks_kernel picks, for every run of 32 pixels of a row, the KW-label range [g0, g0+KW) that
// holds the most windows (the others go to the list), and groups the rows of a block of 32 x 8
// whose ranges lie within KWT labels [G0, G0+KWT) into a task.  Neighbouring rows have nearly the
// same ranges: on the 9x9 x 512^2 light field KWT = 40 takes 1.03 tasks per block (36: 1.50), so
// eight rows share the tiles and the descriptor of one label range.
//
// One CTA of eight warps runs a task, a warp a row, lane = pixel, its KW partial sums in registers.
// Per view the CTA shares one TMA tile of the padded view and one of the padded census words
// (edge-replicated padding: a read at a padded position equals the clamped read); each distinct g0 of
// its rows has a bulk-copied descriptor.  They go through a ring of stages on full / empty mbarriers;
// the warps take turns issuing the refills.  Waits are bounded: on expiry LFSGM_ERR_TIMEOUT is latched.
//
// What bounds it: issue slots and the latency of the segments' dependent steps.  A range splits into
// segments at the labels where the bilinear cell (integer shift) changes; inside a segment the
// fractional shift grows linearly with the label, so the sample minus I_ref(p) is a quadratic
// A + i (B + i Q) in the label index i.  Per (warp, view) the segments' coefficients and the census
// steps cost a fixed number of instructions and the labels three per pixel (two FMAs, one |.|-add).
// The labels are unrolled once, in blocks (grey six, colour one): a segment enters the unrolled code
// at its first block (a switch) and leaves it after its last; a block shared by two segments is
// evaluated by both, each adding its own labels (predicated).  So the coefficients stay in registers.
//
// The census term is a step function of the label: the changes of the Hamming distance at the
// nearest-shift breakpoints are added to a difference column in shared memory (a word holds two
// labels' 16-bit changes) and prefix-summed once at the end.  The finished rows go through shared
// memory so that a window's costs are written side by side.
//
// Colour (C = 3, Sec. III-B/C): float4 pixels (channels interleaved, 4-D tensor map) and the view's
// three census planes; a segment holds the three channels' coefficients, a label's l2 term is the
// Euclidean norm of its three sample differences.  Pixels whose differences leave the range of the fast root
// are appended to the list.
//
// A pixel's costs depend on its row's own g0 only, not on the task that its row is in, and the views
// are added in order.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "lfsgm_internal.cuh"

namespace lfsgm {
namespace {

constexpr int kBlkH = 8, kRowWarps = 8;       // block rows, warps per CTA (a row each)

struct RowPlan {
    int P, Wp, Hp;                    // padding and padded sizes
    int bwf, bhf, bwc, bhc;           // TMA boxes (elements): view values, census words
    int seg_cap;                      // most segments (and census breakpoints) in one label range
    int ds_stride;                    // bytes of one (view, g0) descriptor slot
    int stages, stage;                // ring depth and bytes of a stage: view tile, census tile, descriptors
    int o_rc, o_ds;                   // census tile and the rows' descriptors within a stage
    int o_cd, cd_bytes, o_mbar;       // per-warp difference columns (then output rows), mbarriers
    int o_hd, o_nb;                   // the views' tile headers, their descriptors' sizes (a byte per row, in 16 bytes)
    int smem;                         // shared memory of a CTA
    int kw, kwt;                      // label spans of a row's range (a kernel instantiation) and of a task's
    int C;                            // channels: 1, or 3 (float4 view tiles, three census planes)
};

// Tile header of the labels [G0, G0+kwt) of one view (build_fine_rows_desc), 16 bytes: int16 xf, yf,
// xc, yc, the tile origins relative to (x0, y0); int offsets in the view and census tiles of the
// block's first pixel at shift 0.
// Descriptor of the label range [g0, g0+KW) of one view: what does not depend on the row.
//   bytes  0..15  float ax, ay (the view's (u-uc) * step and (v-vc) * step), ax * ay; uint8 segments,
//                 census steps, uint16 bytes of this descriptor (a multiple of 16)
//   then          per segment 32 bytes: int tile offset of its shift (oy * bwf + ox), int first label |
//                 end label << 16, float fx, fy, fx*fy, fx*ay + fy*ax at the first label, first label
//                 fi, -2 fi
//   then          per census step 16 bytes: int byte offset of its shift, byte offset of its difference
//                 word (label / 2) * 128, shift 16 * (label & 1), 0
constexpr int kDsSegs = 16, kDsSegBytes = 32, kDsCenBytes = 16;

// Bits pos .. pos + len - 1 (past bit 31: none).
__device__ __forceinline__ unsigned bit_mask(int pos, int len) {
    unsigned r;
    asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(r) : "r"(pos), "r"(len));
    return r;
}

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Bounded wait on an mbarrier phase: each try_wait may suspend the thread for up to 200 ns (a hint;
// it returns as soon as the phase completes), so a wait polls a few times instead of spinning, and
// 2^20 tries bound it to about 0.2 s.
__device__ __forceinline__ bool mbar_wait(unsigned mbar, unsigned parity) {
    for (int it = 0; it < (1 << 20); it++) {
        unsigned done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(mbar), "r"(parity), "n"(200) : "memory");
        if (done) return true;
    }
    return false;
}

// One CTA per block of 32 x 8 pixels, a warp per row: every row's range (the start, of its windows'
// starts, whose kw labels hold the most of them; ties: the lowest), then the tasks of the block.  Task
// b (b < nblk) is block b's first (no pixels: none); further ones take the slots from nblk on (*extra
// of them; at most eight tasks a block).  Rows are grouped greedily: the start G0 whose kwt labels hold the
// most pending rows, `most` of them at most.  Wide windows and those outside their row's range go to the list, in
// 32-label chunks.
__global__ void __launch_bounds__(32 * kBlkH) row_tasks_kernel(const int *__restrict__ lo, const int *__restrict__ cnt,
                                                               const long long *__restrict__ off, int G, int H, int W,
                                                               int kw, int kwt, int most, int nblk, RowTask *__restrict__ tasks,
                                                               int *__restrict__ extra, int2 *__restrict__ list,
                                                               int *__restrict__ list_count, int *__restrict__ status,
                                                               const int *__restrict__ large,
                                                               unsigned char *__restrict__ marks) {
    __shared__ int sg0[kBlkH], shi[kBlkH];
    __shared__ unsigned sm[kBlkH];
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
    const int b = blockIdx.x, bx = (W + 31) >> 5;
    const int x = (b % bx) * 32 + lane, y = (b / bx) * kBlkH + r;
    int l = 0, n = 0;
    bool nar = false, todo = false;                       // a narrow window; one for the list
    if (x < W && y < H) {
        const size_t p = (size_t)y * W + x;
        l = __ldg(lo + p);
        n = __ldg(cnt + p);
        if (window_ok(l, n, G, __ldg(off + p + 1) - __ldg(off + p), status)) {
            nar = n <= 32;
            todo = !nar;
        }
    }
    if (marks && y < H) {                                 // warp-uniform
        // a run of whole-range windows (wider than 32 labels) for census_runs
        const bool whole = x >= W || (todo && l == 0 && n == G);
        const bool all = __ballot_sync(0xffffffffu, whole) == 0xffffffffu && !__ldg(large);
        if (lane == 0) marks[(size_t)y * bx + b % bx] = all;
        if (all) todo = false;
    }
    unsigned left = __ballot_sync(0xffffffffu, nar);
    int best = 0, g0 = 0;
    while (left) {
        const int c = __shfl_sync(0xffffffffu, l, __ffs(left) - 1);
        left &= ~__ballot_sync(0xffffffffu, nar && l == c);
        const int fit = __popc(__ballot_sync(0xffffffffu, nar && l >= c && l + n <= c + kw));
        if (fit > best || (fit == best && c < g0)) {
            best = fit;
            g0 = c;
        }
    }
    const bool in = nar && l >= g0 && l + n <= g0 + kw;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    const int hi = (int)__reduce_max_sync(0xffffffffu, in ? (unsigned)(l + n) : 0u);
    if (lane == 0) {
        sg0[r] = g0;
        shi[r] = hi;
        sm[r] = m;
    }
    __syncthreads();
    if (r == 0) {
        // lanes 0 .. 7: a row each
        const int q = lane & (kBlkH - 1);
        const int qg = sg0[q], qh = shi[q];
        const unsigned qm = sm[q];
        unsigned pend = __ballot_sync(0xffffffffu, lane < kBlkH && qm != 0);
        for (int k = 0; k < kBlkH; k++) {
            // the rows that [qg, qg + kwt) holds, if row q is pending; most rows, then the lowest start
            unsigned set = 0;
#pragma unroll
            for (int i = 0; i < kBlkH; i++) {
                const int ig = __shfl_sync(0xffffffffu, qg, i), ih = __shfl_sync(0xffffffffu, qh, i);
                if ((pend >> i & 1) && ig >= qg && ih <= qg + kwt) set |= 1u << i;
            }
            const bool cand = lane < kBlkH && (pend >> lane & 1);
            const unsigned key = cand ? ((unsigned)__popc(set) << 16 | (0xffffu - (unsigned)qg)) : 0u;
            const unsigned top = __reduce_max_sync(0xffffffffu, key);
            if (top == 0) {
                if (k == 0 && lane < kBlkH) tasks[b].mask[lane] = 0;
                break;
            }
            const int src = __ffs(__ballot_sync(0xffffffffu, cand && key == top)) - 1;
            const int G0 = __shfl_sync(0xffffffffu, qg, src);
            set = __shfl_sync(0xffffffffu, set, src);
            while (__popc(set) > most) set &= ~(1u << (31 - __clz(set)));
            int slot = b;
            if (k > 0) {
                slot = nblk;
                if (lane == 0) slot += atomicAdd(extra, 1);
                slot = __shfl_sync(0xffffffffu, slot, 0);
            }
            if (lane < kBlkH) {
                const bool takes = set >> lane & 1;
                tasks[slot].mask[lane] = takes ? qm : 0u;
                tasks[slot].row[lane] = (unsigned char)(takes ? qg - G0 : 0);
            }
            if (lane == 0) {
                tasks[slot].block = b;
                tasks[slot].g0 = G0;
            }
            pend &= ~set;
        }
    }
    todo |= nar && !in;
    // one place in the list per warp
    const int nch = todo ? (n + 31) >> 5 : 0;
    const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)nch);
    if (total == 0) return;
    int incl = nch;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
    }
    int base = lane == 0 ? atomicAdd(list_count, total) : 0;
    base = __shfl_sync(0xffffffffu, base, 0) + incl - nch;
    for (int c = 0; c < nch; c++) list[base + c] = make_int2(y * W + x, c);
}

template <int KW, int C>
__global__ void __launch_bounds__(32 * kRowWarps, 3)
    fine_cost_rows(const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_c,
                   const unsigned char *__restrict__ desc, const int4 *__restrict__ heads,
                   const RowTask *__restrict__ tasks, const int *__restrict__ extra, int nblk, int G, int nviews, int H,
                   int W, int ref, const int *__restrict__ lo, const int *__restrict__ cnt,
                   const long long *__restrict__ off, const float *__restrict__ views_pad,
                   const uint64_t *__restrict__ cen_pad, float wl2, float wc, float *__restrict__ cost,
                   int *__restrict__ status, int2 *__restrict__ list, int *__restrict__ list_count,
                   const __grid_constant__ RowPlan pl) {
    static_assert(KW > 32 && KW <= 44 && KW % 4 == 0, "a range holds every window of at most 32 labels");
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned mbar = smem_u32(smem + pl.o_mbar);      // full[stages] at +0, empty[stages] at +64
    volatile int *gave_up = (volatile int *)(smem + pl.o_mbar + 120);   // a warp's wait has expired
    const int S = pl.stages, ls = S == 4 ? 2 : 1;          // a power of two: view vi uses stage vi mod S
    // a CTA per block and per further task; more than that (the rows of many blocks differ) in turn
    bool inited = false;
    for (int t = blockIdx.x; t < nblk + min(__ldg(extra), (kBlkH - 1) * nblk); t += gridDim.x) {
    const RowTask *task = tasks + t;
    const unsigned any = __ldg(task->mask + (lane & 7));
    if (__ballot_sync(0xffffffffu, any != 0) == 0) continue;           // the whole CTA
    const unsigned mk = __shfl_sync(0xffffffffu, any, w);
    const int blk = __ldg(&task->block), G0 = __ldg(&task->g0);
    // lanes 0 .. 7: the rows' range starts from G0, and the first row with the same one (whose descriptor it uses)
    const int grow = __ldg(task->row + (lane & 7));
    const int lead = __ffs(__match_any_sync(0xffffffffu, any ? grow : 256 + lane)) - 1;
    const int bx = (W + 31) >> 5;
    const int by = blk / bx, x0 = (blk - by * bx) << 5, y0 = by * kBlkH;
    const int x = x0 + lane, y = y0 + w;
    const size_t HWp = (size_t)pl.Hp * pl.Wp;
    const int nv = nviews - 1;                             // the views without the reference
    int4 *hds = (int4 *)(smem + pl.o_hd);
    unsigned char *nbs = smem + pl.o_nb;
    if (inited) {
        __syncthreads();                      // every warp is done with the previous task
        if (*gave_up) return;                 // all of them: the barriers of a warp that gave up are not set up anew
    }
    if (threadIdx.x == 0) {
        if (!inited) *gave_up = 0;
        for (int s = 0; s < S; s++) {
            if (inited) {
                asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mbar + 8 * s) : "memory");
                asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mbar + 64 + 8 * s) : "memory");
            }
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar + 8 * s) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar + 64 + 8 * s), "n"(kRowWarps) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    inited = true;
    // the views' tile headers and the sizes of the rows' descriptors
    for (int i = threadIdx.x; i < nv; i += 32 * kRowWarps) hds[i] = __ldg(heads + (size_t)(i + (i >= ref)) * G + G0);
    for (int i = threadIdx.x; i < 8 * nv; i += 32 * kRowWarps) {
        const int vi = i >> 3, r = i & 7;                  // (r = lane & 7)
        const unsigned char *d = desc + ((size_t)(vi + (vi >= ref)) * G + G0 + grow) * pl.ds_stride;
        nbs[i] = lead == r && any ? (unsigned char)min((unsigned)__ldg(reinterpret_cast<const unsigned short *>(d) + 7) >> 4,
                                                       (unsigned)pl.ds_stride >> 4)
                                  : (unsigned char)0;
    }
    // the lane's pixel: reference values and census words; the warp's labels [j0, j1) from its g0
    const bool on = mk >> lane & 1;
    const int gw = __shfl_sync(0xffffffffu, grow, w), dslot = __shfl_sync(0xffffffffu, lead, w);
    float Iref[C];
    uint64_t cr[C];
    int j0 = 255, j1 = 0;
#pragma unroll
    for (int ch = 0; ch < C; ch++) {
        Iref[ch] = 0.f;
        cr[ch] = 0;
    }
    if (on) {
        const size_t p = (size_t)y * W + x, pp = (size_t)(y + pl.P) * pl.Wp + (x + pl.P);
        j0 = __ldg(lo + p) - G0 - gw;
        j1 = j0 + __ldg(cnt + p);
        if constexpr (C == 1) {
            Iref[0] = __ldg(views_pad + (size_t)ref * HWp + pp);
        } else {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(views_pad) + (size_t)ref * HWp + pp);
            Iref[0] = v.x;
            Iref[1] = v.y;
            Iref[2] = v.z;
        }
#pragma unroll
        for (int ch = 0; ch < C; ch++) cr[ch] = __ldg(cen_pad + ((size_t)ref * C + ch) * HWp + pp);
    }
    j0 = (int)__reduce_min_sync(0xffffffffu, (unsigned)j0);
    j1 = min(KW, (int)__reduce_max_sync(0xffffffffu, (unsigned)j1));
    int *cdw = (int *)(smem + pl.o_cd + w * pl.cd_bytes) + lane;   // [KW / 2][32]: two labels' census steps
#pragma unroll
    for (int i = 0; i < KW / 2; i++) cdw[32 * i] = 0;
    float acc[KW];
#pragma unroll
    for (int i = 0; i < KW; i++) acc[i] = 0.f;
    __syncthreads();

    const unsigned tile_bytes = (unsigned)(pl.bwf * pl.bhf * 4 * (C == 1 ? 1 : 4) + pl.bwc * pl.bhc * 8 * C);
    auto issue = [&](int vi, int st) {                     // one warp
        const int view = vi + (vi >= ref);
        const unsigned nb = lane < 8 ? 16u * nbs[8 * vi + lane] : 0u;
        const unsigned bytes = tile_bytes + __reduce_add_sync(0xffffffffu, nb);
        const unsigned mb = mbar + 8 * st, base = smem_u32(smem) + (unsigned)(st * pl.stage);
        if (lane == 0) {
            const int4 hd = hds[vi];
            const int xf = x0 + (int)(short)(hd.x & 0xffff), yf = y0 + (hd.x >> 16);
            const int xc = x0 + (int)(short)(hd.y & 0xffff), yc = y0 + (hd.y >> 16);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
            if constexpr (C == 1)
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                             ::"r"(base), "l"((unsigned long long)&tm_v), "r"(xf), "r"(yf), "r"(view), "r"(mb) : "memory");
            else                                           // {channel, x, y, view} of the float4 pixels
                asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                             ::"r"(base), "l"((unsigned long long)&tm_v), "r"(0), "r"(xf), "r"(yf), "r"(view), "r"(mb) : "memory");
            asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                         ::"r"(base + pl.o_rc), "l"((unsigned long long)&tm_c), "r"(xc), "r"(yc), "r"(view * C), "r"(mb) : "memory");
        }
        __syncwarp();                                      // (the expected bytes are announced)
        if (nb)
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(base + pl.o_ds + lane * pl.ds_stride), "l"(desc + ((size_t)view * G + G0 + grow) * pl.ds_stride), "r"(nb), "r"(mb) : "memory");
    };
    // Warp w issues the views vi = w mod 8.  The first S views go out at once; view vi + S - lag refills
    // the stage of view vi - lag at the top of iteration vi (lag 2 leaves the warps a view of slack
    // between each other), once all warps have released it.
    const int lag = ls;
    for (int vi = w; vi < min(nv, S); vi += kRowWarps) issue(vi, vi);
    bool ok = true;
    int vi = 0;
    for (; vi < nv; vi++) {
        if (((vi + S - lag) & (kRowWarps - 1)) == w && vi >= lag && vi + S - lag < nv) {   // warp-uniform
            const int q = vi - lag;                        // its stage, released for the (q / S)-th time
            if (!mbar_wait(mbar + 64 + 8 * (q & (S - 1)), (unsigned)(q >> ls) & 1u)) {
                ok = false;
                break;
            }
            issue(vi + S - lag, q & (S - 1));
        }
        const int st = vi & (S - 1);
        if (!mbar_wait(mbar + 8 * st, (unsigned)(vi >> ls) & 1u)) {
            ok = false;
            break;
        }
        if (mk) {                                          // warp-uniform
            const unsigned char *sb = smem + st * pl.stage, *ds = sb + pl.o_ds + dslot * pl.ds_stride;
            const int4 hdr = *(const int4 *)ds;
            const int2 org = *(const int2 *)((const unsigned char *)(hds + vi) + 8);
            const int nseg = min(hdr.w & 0xff, pl.seg_cap), ncen = min((hdr.w >> 8) & 0xff, pl.seg_cap);
            // census: integer steps at the census breakpoints
            {
                const int4 *ce = (const int4 *)(ds + kDsSegs + nseg * kDsSegBytes);
                const unsigned char *rc = sb + pl.o_rc + 8 * (org.y + w * pl.bwc + lane);
                int prev = 0;
#pragma unroll 1
                for (int b = 0; b < ncen; b++) {
                    const int4 e = ce[b];
                    int h = 0;
#pragma unroll
                    for (int ch = 0; ch < C; ch++)
                        h += __popcll(cr[ch] ^ ((const uint64_t *)(rc + e.x))[ch * pl.bwc * pl.bhc]);
                    atomicAdd((int *)((char *)cdw + e.y), (int)((unsigned)(h - prev) << e.z));
                    prev = h;
                }
            }
            // l2 term: per segment the lane's sample polynomial (minus I_ref) in the label index
            const float ax = __int_as_float(hdr.x), ay = __int_as_float(hdr.y), axay = __int_as_float(hdr.z);
            constexpr int TS = C == 1 ? 1 : 4;             // floats of a tile pixel
            const float *rf = (const float *)sb + TS * (org.x + w * pl.bwf + lane);
#pragma unroll 1
            for (int sgi = 0; sgi < nseg; sgi++) {
                const int4 d0 = *(const int4 *)(ds + kDsSegs + sgi * kDsSegBytes);
                const float4 d1 = *(const float4 *)(ds + kDsSegs + sgi * kDsSegBytes + 16);
                const int js = d0.y & 0xffff, jb = max(js, j0), je = min(d0.y >> 16, j1);
                if (je <= jb) continue;                    // warp-uniform
                const float fx = __int_as_float(d0.z), fy = __int_as_float(d0.w);
                float A[C], B[C], Q[C];
#pragma unroll
                for (int ch = 0; ch < C; ch++) {
                    const float *q = rf + TS * d0.x + ch;
                    const float i00 = q[0], i10 = q[TS], i01 = q[TS * pl.bwf], i11 = q[TS * (pl.bwf + 1)];
                    const float c1 = i10 - i00, c2 = i01 - i00, c3 = (i11 - i01) - c1;
                    // s(t) - I_ref = (c0 - I_ref) + c1 fx + c2 fy + c3 fx fy, fx = fx0 + ax t, fy = fy0 + ay t,
                    // t = i - fi: value a0, slope b0 and curvature Q at t = 0, then in powers of i
                    const float a0 = fmaf(c3, d1.x, fmaf(c2, fy, fmaf(c1, fx, i00 - Iref[ch])));
                    const float b0 = fmaf(c3, d1.y, fmaf(c2, ay, c1 * ax));
                    Q[ch] = c3 * axay;
                    A[ch] = fmaf(d1.z, fmaf(d1.z, Q[ch], -b0), a0);
                    B[ch] = fmaf(d1.w, Q[ch], b0);
                }
                // its labels, LB at a time: enter the unrolled blocks at the first, leave them after the last;
                // labels of a block outside the segment (its mask) are evaluated but not added
                constexpr int LB = C == 1 ? 6 : 1;
                const int ke = (je + LB - 1) / LB;
                const unsigned mask = bit_mask(js, je - js);
                auto block = [&](auto K) {
#pragma unroll
                    for (int e = 0; e < LB; e++) {
                        constexpr int k0 = LB * decltype(K)::value;
                        const int i = k0 + e;
                        const float f = (float)i;
                        float v;
#pragma unroll
                        for (int ch = 0; ch < C; ch++) {
                            const float u = fmaf(f, fmaf(f, Q[ch], B[ch]), A[ch]);
                            if constexpr (C == 1) v = fabsf(u);
                            else v = ch ? fmaf(u, u, v) : u * u;
                        }
                        if constexpr (C > 1) v = sqrt_fast(v);
                        // (labels below 32 by the mask)
                        if (i < KW && (LB == 1 || (i < 32 ? (mask >> (i & 31) & 1) != 0 : i >= js && i < je))) acc[i] += v;
                    }
                };
                switch (jb / LB) {
#define LFSGM_B(k)                                             \
    case k:                                                    \
        if constexpr (LB * (k) < KW) {                         \
            block(std::integral_constant<int, k>{});           \
            if (ke == (k) + 1) break;                          \
        }                                                      \
        [[fallthrough]];
#define LFSGM_B4(k) LFSGM_B(k) LFSGM_B(k + 1) LFSGM_B(k + 2) LFSGM_B(k + 3)
                    LFSGM_B4(0) LFSGM_B4(4) LFSGM_B4(8) LFSGM_B4(12) LFSGM_B4(16) LFSGM_B4(20) LFSGM_B4(24)
                    LFSGM_B4(28) LFSGM_B4(32) LFSGM_B4(36) LFSGM_B4(40)
#undef LFSGM_B4
#undef LFSGM_B
                default: break;
                }
            }
        }
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar + 64 + 8 * st) : "memory");
    }
    if (!ok) {
        if (lane == 0) {
            atomicExch(status, 6);
            *gave_up = 1;
        }
        // let the copies still in flight land (bounded) before the CTA's shared memory is released
        for (int v = vi; v < min(nv, vi + S); v++) mbar_wait(mbar + 8 * (v & (S - 1)), (unsigned)(v >> ls) & 1u);
    }
    if (!ok || mk == 0) continue;                          // (to the barrier above)
    if constexpr (C > 1) {
        // sqrt_fast's range: a squared difference that overflows gives NaN, one below 2^-126 is off by at most
        // 2^-63.  A pixel with a sum that is not finite, or not 0 and so small that this shows, goes to the list
        // kernel, which runs next and takes sqrtf.  (Looking at each segment's coefficients for it: 2377 -> 2464 us
        // on the 9x9 x 512^2 final map; here, once per pixel, within 0.1 %.)
        bool redo = false;
#pragma unroll
        for (int i = 0; i < KW; i++) redo |= !(acc[i] < __int_as_float(0x7f800000)) || (acc[i] > 0.f && acc[i] < 0x1p-29f);
        const unsigned rm = __ballot_sync(0xffffffffu, redo && on);
        if (rm) {
            int base = lane == 0 ? atomicAdd(list_count, __popc(rm)) : 0;
            base = __shfl_sync(0xffffffffu, base, 0);
            if (rm >> lane & 1) list[base + __popc(rm & ((1u << lane) - 1u))] = make_int2(y * W + x, 0);
        }
    }
    // a word holds d(i) + d(i+1) 2^16 (two's complement, |d| < 2^15): split it exactly
    int run = 0;
#pragma unroll
    for (int i = 0; i < KW; i += 2) {
        const int dw = cdw[16 * i];
        const int d0 = (int)(short)(dw & 0xffff);
        run += d0;
        acc[i] = fmaf(wc, (float)run, wl2 * acc[i]);
        run += (dw - d0) >> 16;
        acc[i + 1] = fmaf(wc, (float)run, wl2 * acc[i + 1]);
    }
    // the pixels through shared memory, 16 at a time (row stride KW + 1: no bank conflicts), each window
    // then written by the warp side by side, its padding slots with 0
    float *tb = (float *)(smem + pl.o_cd + w * pl.cd_bytes);
    int ln = 0, np = 0;
    long long o = 0;
    if (on) {
        const size_t p = (size_t)y * W + x;
        const int n = __ldg(cnt + p);
        ln = (__ldg(lo + p) - G0 - gw) | (n << 16);
        o = __ldg(off + p);
        np = (int)min((long long)((n + 3) & ~3), __ldg(off + p + 1) - o);
    }
#pragma unroll
    for (int hf = 0; hf < 2; hf++) {
        __syncwarp();
        if ((lane >> 4) == hf) {
#pragma unroll
            for (int i = 0; i < KW; i++) tb[(lane & 15) * (KW + 1) + i] = acc[i];
        }
        __syncwarp();
#pragma unroll 4
        for (int q = 0; q < 16; q++) {
            const int lnq = __shfl_sync(0xffffffffu, ln, 16 * hf + q), npq = __shfl_sync(0xffffffffu, np, 16 * hf + q);
            const long long oq = __shfl_sync(0xffffffffu, o, 16 * hf + q);
            if (lane < npq) cost[oq + lane] = lane < (lnq >> 16) ? tb[q * (KW + 1) + (lnq & 0xffff) + lane] : 0.f;
        }
    }
    }
}

int r128(int x) { return (x + 127) & ~127; }

}  // namespace

int row_blocks(int H, int W) { return ((W + 31) / 32) * ((H + kBlkH - 1) / kBlkH); }

// Padding, TMA boxes and the shared-memory layout of the row kernel for one config.
bool plan_fine_rows(int U, int V, int uc, int vc, int H, int W, int G, double dmin, double dmax, int kw, int C,
                    RowPlanHost *out) {
    RowPlan pl{};
    const int kRowKW = kw == 44 ? 44 : 36;
    pl.kw = kRowKW;
    pl.C = C;
    const double md = fmax(fabs(dmin), fabs(dmax));
    const int amax = std::max(std::max(uc, U - 1 - uc), std::max(vc, V - 1 - vc));
    pl.P = (int)ceil(amax * md) + 3;
    pl.Wp = (W + 2 * pl.P + 3) & ~3;
    pl.Hp = H + 2 * pl.P;
    const double step = (dmax - dmin) / (double)(G - 1);
    const int ax = std::max(uc, U - 1 - uc), ay = std::max(vc, V - 1 - vc);
    // a task spans 4 labels more than a row's range, or, where a box would then be too large for TMA, none
    for (int more = 4; more >= 0; more -= 4) {
        pl.kwt = kRowKW + more;
        const int spx = (int)ceil(ax * step * (pl.kwt - 1)), spy = (int)ceil(ay * step * (pl.kwt - 1));
        // taps: columns x0+oxlo .. x0+32+oxhi, rows y0+oylo .. y0+7+oyhi+1, with oxhi-oxlo <= spx, one label of
        // slack below the FP32 origin estimate and up to 3 (floats) / 1 (words) columns of 16-byte rounding
        pl.bwf = (spx + 38 + 3) & ~3;
        pl.bhf = spy + 4 + kBlkH - 1;
        pl.bwc = (spx + 35 + 1) & ~1;
        pl.bhc = spy + 3 + kBlkH - 1;
        if (pl.bwf <= 256 && pl.bwc <= 256 && pl.bhf <= 256 && pl.bhc <= 256) break;
    }
    pl.seg_cap = std::min(kRowKW, (int)ceil(ax * step * (kRowKW - 1)) + (int)ceil(ay * step * (kRowKW - 1)) + 3);
    pl.ds_stride = (kDsSegs + pl.seg_cap * (kDsSegBytes + kDsCenBytes) + 15) & ~15;
    pl.o_rc = r128(pl.bwf * pl.bhf * 4 * (C == 1 ? 1 : 4));               // colour: float4 pixels
    pl.o_ds = pl.o_rc + r128(pl.bwc * pl.bhc * 8 * C);                    // one plane per channel
    pl.stage = r128(pl.o_ds + kBlkH * pl.ds_stride);
    pl.cd_bytes = r128(std::max(kRowKW / 2 * 128, 16 * (kRowKW + 1) * 4));
    // four stages where they leave room for the three CTAs per SM that the registers allow
    const int rest = kRowWarps * pl.cd_bytes + 128 + 16 * U * V + r128(8 * U * V);
    pl.stages = 4 * pl.stage + rest <= 75 * 1024 ? 4 : 2;
    pl.o_cd = pl.stages * pl.stage;
    pl.o_mbar = pl.o_cd + kRowWarps * pl.cd_bytes;
    pl.o_hd = pl.o_mbar + 128;
    pl.o_nb = pl.o_hd + 16 * U * V;
    pl.smem = pl.o_nb + r128(8 * U * V);
    // Ranges that spread over many pixels (large label steps) take the list kernel: a range of 36 labels
    // over 27 x 27 pixels has a segment per label, so nothing is shared.  The bound is a run's footprint
    // (two view tiles, a census tile, 32 + 48 bytes of descriptor and 384 of coefficients per segment).
    const int fx = (int)ceil(ax * step * (kRowKW - 1)), fy = (int)ceil(ay * step * (kRowKW - 1));
    const int ftile = r128(((fx + 41) & ~3) * (fy + 4) * 4 * (C == 1 ? 1 : 4)), fds = 32 + pl.seg_cap * 48;
    const int footprint = 2 * r128(ftile + fds) + r128(((fx + 36) & ~1) * (fy + 3) * 8 * C) + pl.seg_cap * 384 +
                          kRowKW / 2 * 128 + 32;
    // the census steps of one label, summed over the views and channels, must fit 16 bits (at most 48
    // bits a word); colour runs the 36-label span only
    out->ok = pl.bwf <= 256 && pl.bwc <= 256 && pl.bhf <= 256 && pl.bhc <= 256 && footprint <= 48 * 1024 &&
              pl.smem <= 220 * 1024 &&
              (U * V - 1) * 48 * C < 32768 && pl.ds_stride <= 255 * 16 && (C == 1 || (C == 3 && kRowKW == 36));
    static_assert(sizeof(RowPlan) <= sizeof(out->raw), "plan storage");
    memcpy(out->raw, &pl, sizeof(pl));
    out->P = pl.P;
    out->Wp = pl.Wp;
    out->Hp = pl.Hp;
    return out->ok;
}

// Tile headers and descriptors of every (view, g0) label range for the row kernel, from the host copy
// of the tap table.  The tile origins follow an FP32 estimate of the shifts (one label of slack around
// the range's shifts, x rounded down to 16 bytes); every tap and census word of the range is
// checked to lie inside the tile boxes here, so the kernel needs no bounds test.  Returns false
// (the caller then sends every window to the list kernel) if any range does not fit.
bool build_fine_rows_desc(const RowPlanHost *ph, const FineTap *tab, int U, int V, int uc, int vc, int G, float dmin,
                          float fstep, std::vector<unsigned char> &out, std::vector<int4> &heads) {
    RowPlan pl;
    memcpy(&pl, ph->raw, sizeof(pl));
    const int nviews = U * V;
    const size_t bytes = (size_t)nviews * G * pl.ds_stride;
    if (bytes > ((size_t)512 << 20)) return false;
    out.assign(bytes, 0);
    heads.assign((size_t)nviews * G, make_int4(0, 0, 0, 0));
    std::vector<int> segstart, censtart;
    for (int view = 0; view < nviews; view++) {
        const float a = (float)(view % U - uc), b = (float)(view / U - vc);
        for (int g0 = 0; g0 < G; g0++) {
            const FineTap *t = tab + (size_t)view * G + g0;
            {   // the tiles of the labels [g0, g0 + kwt)
                const int nvalid = std::min(pl.kwt, G - g0);
                const float d0 = std::fmaf((float)g0, fstep, dmin), d1 = std::fmaf((float)(g0 + nvalid - 1), fstep, dmin);
                const float sx0 = a * d0, sx1 = a * d1, sy0 = b * d0, sy1 = b * d1;
                const int xf = ((int)std::floor(std::fmin(sx0, sx1)) - 1 + pl.P) & ~3;
                const int yf = (int)std::floor(std::fmin(sy0, sy1)) - 1 + pl.P;
                const int xc = ((int)std::floor(std::fmin(sx0, sx1) + 0.5f) - 1 + pl.P) & ~1;
                const int yc = (int)std::floor(std::fmin(sy0, sy1) + 0.5f) - 1 + pl.P;
                const int bxf = pl.P - xf, byf = pl.P - yf, bxc = pl.P - xc, byc = pl.P - yc;
                int oxlo = 1 << 30, oxhi = -(1 << 30), oylo = 1 << 30, oyhi = -(1 << 30);
                int nxlo = 1 << 30, nxhi = -(1 << 30), nylo = 1 << 30, nyhi = -(1 << 30);
                for (int i = 0; i < nvalid; i++) {
                    oxlo = std::min(oxlo, (int)t[i].ox);
                    oxhi = std::max(oxhi, (int)t[i].ox);
                    oylo = std::min(oylo, (int)t[i].oy);
                    oyhi = std::max(oyhi, (int)t[i].oy);
                    nxlo = std::min(nxlo, (int)t[i].nx);
                    nxhi = std::max(nxhi, (int)t[i].nx);
                    nylo = std::min(nylo, (int)t[i].ny);
                    nyhi = std::max(nyhi, (int)t[i].ny);
                }
                constexpr int last = kBlkH - 1;          // the block's last row
                if (bxf + oxlo < 0 || bxf + 32 + oxhi >= pl.bwf || byf + oylo < 0 || byf + oyhi + 1 + last >= pl.bhf ||
                    bxc + nxlo < 0 || bxc + 31 + nxhi >= pl.bwc || byc + nylo < 0 || byc + nyhi + last >= pl.bhc)
                    return false;
                heads[(size_t)view * G + g0] = make_int4((xf & 0xffff) | yf << 16, (xc & 0xffff) | yc << 16,
                                                         byf * pl.bwf + bxf, byc * pl.bwc + bxc);
            }
            const int nvalid = std::min(pl.kw, G - g0);
            segstart.clear();
            censtart.clear();
            for (int i = 0; i < nvalid; i++) {
                if (i == 0 || t[i].ox != t[i - 1].ox || t[i].oy != t[i - 1].oy) segstart.push_back(i);
                if (i == 0 || t[i].nx != t[i - 1].nx || t[i].ny != t[i - 1].ny) censtart.push_back(i);
            }
            const int nseg = (int)segstart.size(), ncen = (int)censtart.size();
            if (nseg > pl.seg_cap || ncen > pl.seg_cap) return false;
            unsigned char *d = out.data() + ((size_t)view * G + g0) * pl.ds_stride;
            // the view's disparity-to-shift factors (u-uc) * step, (v-vc) * step and their product
            const float ax = a * fstep, ay = b * fstep;
            const float axy[3] = {ax, ay, ax * ay};
            memcpy(d, axy, 12);
            d[12] = (unsigned char)nseg;
            d[13] = (unsigned char)ncen;
            const uint16_t nbytes = (uint16_t)(kDsSegs + nseg * kDsSegBytes + ncen * kDsCenBytes);
            memcpy(d + 14, &nbytes, 2);
            for (int k = 0; k < nseg; k++) {
                const FineTap &w = t[segstart[k]];
                unsigned char *e = d + kDsSegs + k * kDsSegBytes;
                const int je = k + 1 < nseg ? segstart[k + 1] : nvalid;
                const int32_t d0[2] = {(int)w.oy * pl.bwf + (int)w.ox, segstart[k] | je << 16};
                const float f[6] = {w.fx, w.fy, w.fx * w.fy, std::fmaf(w.fx, ay, w.fy * ax), (float)segstart[k],
                                    -2.f * (float)segstart[k]};
                memcpy(e, d0, 8);
                memcpy(e + 8, f, 24);
            }
            for (int k = 0; k < ncen; k++) {
                const FineTap &w = t[censtart[k]];
                const int32_t e4[4] = {8 * ((int)w.ny * pl.bwc + (int)w.nx), (censtart[k] >> 1) * 128,
                                       16 * (censtart[k] & 1), 0};
                memcpy(d + kDsSegs + nseg * kDsSegBytes + k * kDsCenBytes, e4, 16);
            }
        }
    }
    return true;
}

// Tensor maps of the padded views (float) and census words (uint64), 3-D [view][Hp][Wp].
bool encode_fine_rows_maps(RowPlanHost *ph, const float *views_pad, const uint64_t *cen_pad, int nviews) {
    RowPlan pl;
    memcpy(&pl, ph->raw, sizeof(pl));
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void *fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return false;
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    if (pl.C == 3) {
        // float4 pixels (the fourth float is padding): {channel, x, y, view}
        const cuuint64_t dims[4] = {4, (cuuint64_t)pl.Wp, (cuuint64_t)pl.Hp, (cuuint64_t)nviews};
        const cuuint64_t strides[3] = {16, (cuuint64_t)pl.Wp * 16, (cuuint64_t)pl.Wp * pl.Hp * 16};
        const cuuint32_t box[4] = {4, (cuuint32_t)pl.bwf, (cuuint32_t)pl.bhf, 1};
        if (encode((CUtensorMap *)ph->tm_v, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void *)views_pad, dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    } else {
        const cuuint64_t dims[3] = {(cuuint64_t)pl.Wp, (cuuint64_t)pl.Hp, (cuuint64_t)nviews};
        const cuuint64_t strides[2] = {(cuuint64_t)pl.Wp * 4, (cuuint64_t)pl.Wp * pl.Hp * 4};
        const cuuint32_t box[3] = {(cuuint32_t)pl.bwf, (cuuint32_t)pl.bhf, 1};
        if (encode((CUtensorMap *)ph->tm_v, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void *)views_pad, dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    {
        // census planes view * C + c: a view's C planes are one box of depth C
        const cuuint64_t dims[3] = {(cuuint64_t)pl.Wp, (cuuint64_t)pl.Hp, (cuuint64_t)nviews * pl.C};
        const cuuint64_t strides[2] = {(cuuint64_t)pl.Wp * 8, (cuuint64_t)pl.Wp * pl.Hp * 8};
        const cuuint32_t box[3] = {(cuuint32_t)pl.bwc, (cuuint32_t)pl.bhc, (cuuint32_t)pl.C};
        if (encode((CUtensorMap *)ph->tm_c, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, (void *)cen_pad, dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
    }
    return true;
}

// Small images: fewer rows a task, so that the tasks are spread over the 152 SMs (up to two on each), instead of eight
// busy warps on few of them.  us, eight rows / up to 152 tasks / 304 / 456: 9x9 x 51 x 87 (21 blocks) 253, 219, 228, 228 (a
// warp per row with its own tile: 227); 9x9 x 160 x 192 (120 blocks) 156, 158, 140, 140; 9x9 x 64^2 in colour 313, 270, 270, 270;
// 15x15 x 104 x 89 (39 blocks) 919, 826, 846, 1555 (704); 15x15 x 128^2 (64 blocks) 322, 342, 348, 350 (407).
static int rows_a_task(int nblk) {
    int rows = kBlkH;
    while (rows > 1 && kBlkH / rows * nblk * 2 <= 304) rows /= 2;
    return rows;
}

cudaError_t launch_row_tasks(cudaStream_t s, const RowPlanHost *ph, int G, int H, int W, const int *lo, const int *cnt,
                             const long long *off, RowTask *tasks, int *extra, int *status, int2 *list,
                             int *list_count, const int *large, unsigned char *marks) {
    RowPlan pl;
    memcpy(&pl, ph->raw, sizeof(pl));
    const int nblk = row_blocks(H, W);
    row_tasks_kernel<<<nblk, 32 * kBlkH, 0, s>>>(lo, cnt, off, G, H, W, pl.kw, pl.kwt, rows_a_task(nblk), nblk, tasks, extra, list, list_count,
                                                    status, large, marks);
    return cudaGetLastError();
}

cudaError_t launch_fine_cost_rows(cudaStream_t s, const RowPlanHost *ph, const float *views_pad,
                                  const uint64_t *cen_pad, const unsigned char *desc, const int4 *heads,
                                  const RowTask *tasks, const int *extra, int G, int nviews, int H, int W, int ref, const int *lo,
                                  const int *cnt, const long long *off, float wl2, float wc, float *cost, int *status,
                                  int2 *list, int *list_count) {
    RowPlan pl;
    memcpy(&pl, ph->raw, sizeof(pl));
    auto kern = pl.C == 3 ? fine_cost_rows<36, 3> : (pl.kw == 44 ? fine_cost_rows<44, 1> : fine_cost_rows<36, 1>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, pl.smem);
    if (e != cudaSuccess) return e;
    // a CTA per block and, for further tasks, as many again (small images, whose blocks often need
    // several: up to one for every possible task); the rest take turns
    const int nblk = row_blocks(H, W), more = std::min(7 * nblk, std::max(nblk, 608));
    kern<<<nblk + more, 32 * kRowWarps, pl.smem, s>>>(*(const CUtensorMap *)ph->tm_v, *(const CUtensorMap *)ph->tm_c, desc,
                                                  heads, tasks, extra, nblk, G, nviews, H, W, ref, lo, cnt, off,
                                                  views_pad, cen_pad, wl2, wc, cost, status, list, list_count, pl);
    return cudaGetLastError();
}

}  // namespace lfsgm

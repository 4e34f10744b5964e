// k_sgm.cu -- bounded SGM over 8 or 16 paths on the windowed fine cost (Sec. III-E with Eq. 8-9).
//
// One warp per (direction, scanline).  Lane j owns slot j of the current pixel's window.
// When this window and the predecessor's are both at most 32 labels wide (the regular case),
// the predecessor's path costs L' stay in registers, one slot per lane, and the ragged-window
// alignment (slot i = lo(p) + j - lo(p-r)) is three shuffles with bounds checks: labels outside
// the predecessor's window are absent from the minimum (Sec. III-E).  Wider windows take the
// general form with L' in a per-warp shared-memory row (chunks of 32 slots).  Window metadata
// is fetched 32 pixels at a time (one per lane, the next block one block ahead) and also kept in a
// per-warp ring of 64 steps in shared memory; a ballot over a block finds the steps that need the
// general form, and the narrow steps between them run in a tight loop that reads the metadata of
// the step after next from the ring (one broadcast load) and loads cost rows two steps ahead.
// The step is the normalised recurrence
//   L(p,g) = C(p,g) + (min(L'(g), L'(g-1)+P1, L'(g+1)+P1, m+P2) - m),   m = min L',
// and the predecessor minimum m is one redux.sync.min.f32 per pixel.  The 8 or 16 directions run
// concurrently and add into agg (zeroed by the caller) with float atomics.  A run of equal windows of
// 33 to 128 labels (whole-range searches) keeps the predecessor's row in registers, four consecutive
// labels a lane: one vector load and one vector reduction a step, the neighbours across lanes by two
// shuffles (7x1 x 555x650, 121 labels: 295 instructions a step in shared-memory chunks, 956 us).  The few
// scanlines that cross many wide windows (a speed knob's threshold) run on all the warps of a CTA each, which
// share the wide steps (sgm_scanline SPLIT); the kernel before lists them.  Where few windows are wide, a warp
// takes two scanlines (sgm_pair).
//
// What bounds it: issue slots while all scanlines run (72 instructions a narrow step, 100 for two in
// sgm_pair), then the scanlines with the most wide steps, and L2 latency where there are few scanlines.
// fine_sgm of 9x9 x 512^2 (31 labels, 0.8 % wide): 297 us before the split by default and the pairs, 209 now
// (recording, not paired: 382 and 314); 15x15 x 434 x 625 (no wide windows): 182 and 165; 4x4 x 720 x 1280, 16
// directions, 17 labels: 1163 and 800.
//
// Reproducible sum over the directions.  The aggregate C_s(p,g) = sum_r L_r(p,g) must not depend on
// the order in which the directions' atomics arrive.  Every exact L_r(p,g) lies in [0, B] with
// B = C(p,g) + P2 (the bracket is at most P2 above m), and B depends only on the cell.  Each
// direction clamps its FP32 L_r to B (removing rounding beyond the exact bound) and rounds it to a
// multiple of q = 2^(floor(log2 B) + 1 + log2(paths) - 24) before adding it.  Then every partial sum
// is a multiple of q no larger than paths x 2^(floor(log2 B) + 1) = 2^24 q, so it is exactly
// representable: each addition is exact, and the sum is the same in any order.  The rounding moves
// an addend by at most q / 2 <= 2^-21 B (8 paths) or 2^-20 B (16 paths).
//
// Derived penalties: per-block partial sums (double) of the active slots, then one block
// adds the partials in a fixed order, so the mean is deterministic.
#include "lfsgm_internal.cuh"

#include <algorithm>

namespace lfsgm {
namespace {

constexpr int kSgmWarps = 4;      // default warps (scanlines) per CTA; 2, 4 or 8 (a speed knob)
constexpr int kSplitRing = 4;     // cost rows of a split scanline's wide steps on their way (a power of two)
constexpr int kPairFrom = 1024;   // scanlines from which on a warp may take two (twelve 5x5 x 251 x 283 side by side:
                                  // 2015 us with one, 1914 with two; 764 scanlines of 5x5 x 64^2: 20.6 and 21.0)
constexpr int kPairPlaces = 2 * 28 * 152;   // scanlines in flight at once, two a warp
constexpr int kSplitCap = 256;    // most scanlines split across a CTA's warps (more qualify: none is)

// L rounded to a multiple of q (see above); B = C + P2 of the cell.  With M = 1.5 x 2^(floor(log2 B)
// + 23 - qsh), qsh = 23 - log2(paths), every x in [0, B] gives x + M in M's binade, whose spacing
// is q: fl(x + M) - M is x rounded to a multiple of q (half to even), and the subtraction is exact.
// mk = (23 - qsh) << 23 | 1 << 22 puts M's exponent and its leading fraction bit in place.
__device__ __forceinline__ float det_addend(float L, float B, int mk) {
    const float M = __int_as_float((__float_as_int(B) & 0x7f800000) + mk);
    return __fsub_rn(__fadd_rn(fminf(L, B), M), M);
}

// agg[0 .. n) to 0 by `stride` threads, this one the i0-th (agg 16-byte aligned).
__device__ __forceinline__ void zero_rows(float *agg, long long n, long long i0, long long stride) {
    const long long n4 = n >> 2;
    float4 *z = reinterpret_cast<float4 *>(agg);
    for (long long i = i0; i < n4; i += stride) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 < (n & 3)) agg[4 * n4 + i0] = 0.f;
}

__device__ __forceinline__ float warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// st.cum[r] by selects (a run-time index would copy the table to the stack).
__device__ __forceinline__ int scan_base(const ScanTable &st, int r) {
    int base = 0;
#pragma unroll
    for (int q = 1; q < kMaxPaths; q++)
        if (q <= r) base = st.cum[q];
    return base;
}

// Four consecutive labels j0 .. j0 + 3 of a wide step on the predecessor's row A by slot (window (pl, pn),
// minimum m; pn = 0: the path starts; same: the windows are equal) with costs c4: the path costs into row
// B (+inf from slot n on) and, rounded, into agg; branches into code; the running minimum and its lowest
// slot (REC) into lmin, lslot.
template <bool REC>
__device__ __forceinline__ void wide_cells(float4 c4, int j0, int n, int l, int pl, int pn, bool same, unsigned top,
                                           const float *A, float m, float P1, float P2, int mk, float *agg,
                                           unsigned char *code, float &lmin, int &lslot, float *B) {
    const float INF = __int_as_float(0x7f800000);
    const float c[4] = {c4.x, c4.y, c4.z, c4.w};
    float v[6], L4[4], a4[4];                  // v: the predecessor's labels -1 .. 4 from j0 on
    unsigned cd = 0u;
    if (same) {
        const float4 f = *reinterpret_cast<const float4 *>(A + j0);
        v[0] = A[j0 - 1];
        v[1] = f.x;
        v[2] = f.y;
        v[3] = f.z;
        v[4] = f.w;
        v[5] = A[j0 + 4];
    } else {
        // slot s is read at A[s] with s + 1 clamped (unsigned) to pn + 1: any slot outside [0, pn) lands on
        // a sentinel (+inf), so an absent label drops out of the minimum
#pragma unroll
        for (int u = 0; u < 6; u++) v[u] = A[(int)min((unsigned)(l + j0 + u - pl), top) - 1];
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const bool on = j0 + u < n;
        const float t = fminf(fminf(m + P2, v[u + 1]), fminf(v[u], v[u + 2]) + P1);
        const float Ln = pn != 0 ? c[u] + (t - m) : c[u];
        if (REC) {
            cd |= (pn == 0 ? 4u : (t == m + P2 ? 3u : (t == v[u + 1] ? 0u : (t == v[u] + P1 ? 1u : 2u)))) << (8 * u);
            if (on && Ln < lmin) lslot = j0 + u;   // ascending: the lane's first minimum
        }
        a4[u] = on ? det_addend(Ln, c[u] + P2, mk) : 0.f;
        L4[u] = on ? Ln : INF;
        lmin = fminf(lmin, L4[u]);
    }
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                 ::"l"(agg + j0), "f"(a4[0]), "f"(a4[1]), "f"(a4[2]), "f"(a4[3]) : "memory");
    if (REC) *reinterpret_cast<unsigned *>(code + j0) = cd;   // the padding slots' codes are never read
    *reinterpret_cast<float4 *>(B + j0) = make_float4(L4[0], L4[1], L4[2], L4[3]);
}

// One scanline of direction r = rs & 15, number s = rs >> 4.  NW = 1: one warp, its own rows by
// slot (bufA, bufB) and metadata ring.  SPLIT (NW = the CTA's warps): the CTA's warps share the
// rows; warp 0 alone runs the narrow steps (the predecessor row in its registers), and every
// general step (a window or predecessor wider than 32 labels, or an invalid window) is spread over
// the warps, four consecutive labels a thread (vectors of cost, aggregate and row; the next step's
// cost one step ahead), the predecessor minimum taken
// over the warps' minima through xm ([2][NW] minima, [2][NW] slots for REC, then the minimum that
// warp 0 hands over after narrow steps), with one CTA barrier per general step (two after narrow
// steps).  Every cell gets the same value either way.
// REC: also record, for the adjoint, each cell's winning branch (0 same label, 1 label-1, 2 label+1,
// 3 m+P2, 4 path start; the first of P2, same, g-1, g+1 that equals the minimum, as the adjoint's
// own recurrence decides it) in codes[r * nnz_cap + slot] (nnz_cap a multiple of 4: vectors of codes) and each pixel's lowest minimising slot
// in amin[r * N + p].
template <bool REC, bool SPLIT, int NW>
__device__ __forceinline__ void sgm_scanline(const float *__restrict__ cost, const int *__restrict__ lo,
                                             const int *__restrict__ cnt, const long long *__restrict__ off,
                                             int H, int W, float P1, float P2, int G, float *__restrict__ agg,
                                             int *__restrict__ status, int rs, int mk,
                                             unsigned char *__restrict__ codes, int *__restrict__ amin,
                                             size_t nnz_cap, float *bufA, float *bufB, int2 *meta, float *xm,
                                             int wib, float *cring = nullptr, int cstride = 0) {
    const int lane = threadIdx.x & 31;
    const int r = rs & 15, s = rs >> 4;
    int dx, dy, x0, y0;
    dir_of(r, dx, dy);
    scan_start_d(dx, dy, s, H, W, x0, y0);
    const int len = scan_steps(x0, y0, dx, dy, H, W);
    unsigned char *code = REC ? codes + (size_t)r * nnz_cap : nullptr;
    int *am = REC ? amin + (size_t)r * H * W : nullptr;
    const float INF = __int_as_float(0x7f800000);
    const bool lead = !SPLIT || wib == 0;        // the warp that runs the narrow steps
    if (SPLIT ? threadIdx.x == 0 : lane == 0) {
        bufA[-1] = INF;
        bufB[-1] = INF;
    }
    const long long p0 = (long long)y0 * W + x0, dpix = (long long)dy * W + dx;
    // window metadata of the 32 steps starting at kb, one step per lane: (lo | cnt << 16) with
    // cnt = 0 for an invalid window, and the row offset in units of 4 slots
    auto fetch = [&](int kb, int &mw, int &mo) {
        const int k = kb + lane;
        mw = 0;
        mo = 0;
        if (k < len) {
            const long long p = p0 + (long long)k * dpix;
            const int l_ = __ldg(lo + p), n_ = __ldg(cnt + p);
            const long long o_ = __ldg(off + p), e_ = __ldg(off + p + 1);   // both multiples of 4: rows end there too
            if (window_ok(l_, n_, G, e_ - o_, status) && ((o_ | e_) & 3) == 0 && (o_ >> 2) < 0x7fffffff) {
                mw = l_ | (n_ << 16);
                mo = (int)(o_ >> 2);
            } else if (((o_ | e_) & 3) != 0 && status) {
                atomicExch(status, 7);
            }
        }
    };
    int cw, co, nw = 0, no = 0;                // this block's and the next block's metadata
    fetch(0, cw, co);
    if (len > 32) fetch(32, nw, no);
    meta[lane] = make_int2(cw, co);
    meta[32 + lane] = make_int2(nw, no);
    if (SPLIT) __syncthreads();                // the sentinels
    else __syncwarp();
    int plo = 0, pn = 0;                       // predecessor window; pn = 0: the path (re)starts
    float prev = INF, m = 0.f;                 // predecessor row (one slot per lane) and its minimum
    bool in_smem = false;                      // the predecessor row is in bufA (after a general step)
    int gpar = 0;                              // SPLIT: which half of xm this general step uses
    int asked = 0;                             // SPLIT: the wide steps before this one are requested (see below)
    int k = 0;
    // the block of metadata after the one that ends at step k (a multiple of 32)
    auto next_block = [&]() {
        cw = nw;
        co = no;
        if (k + 32 < len) {
            fetch(k + 32, nw, no);
        } else {
            nw = 0;
            no = 0;
        }
        meta[(k + 32 + lane) & 63] = make_int2(nw, no);   // the slots of the block just finished
        __syncwarp();
    };
    while (k < len) {
        if constexpr (!REC && !SPLIT) {
            // a run of windows equal to the predecessor's, 33 to 128 labels, after a general step
            if (in_smem && pn > 32 && pn <= 128 && meta[k & 63].x == (plo | (pn << 16))) {
                const int pw = meta[k & 63].x, j0 = 4 * lane;
                // the labels j0 .. j0 + 3 that the window has (the padding slots of a row are never used)
                const bool h0 = j0 < pn, h1 = j0 + 1 < pn, h2 = j0 + 2 < pn, h3 = j0 + 3 < pn;
                float v0 = h0 ? bufA[j0] : INF, v1 = h1 ? bufA[j0 + 1] : INF;
                float v2 = h2 ? bufA[j0 + 2] : INF, v3 = h3 ? bufA[j0 + 3] : INF;
                const float4 *cb = reinterpret_cast<const float4 *>(cost) + lane;
                float *ab = agg + j0;
                const float4 none = make_float4(INF, INF, INF, INF);
                // cost rows two steps ahead; a step that is not in the run loads nothing
                auto row = [&](int2 mt) { return h0 && mt.x == pw ? __ldg(cb + mt.y) : none; };
                int2 mt = meta[k & 63], mt1 = meta[(k + 1) & 63];
                float4 c = row(mt), c1 = row(mt1);
                for (;;) {
                    const int2 mt2 = meta[(k + 2) & 63];
                    const float4 c2 = row(mt2);
                    if (!h1) c.y = INF;
                    if (!h2) c.z = INF;
                    if (!h3) c.w = INF;
                    const float vl = __shfl_up_sync(0xffffffffu, v3, 1), vr = __shfl_down_sync(0xffffffffu, v0, 1);
                    const float left = lane == 0 ? INF : vl, right = lane == 31 ? INF : vr;
                    const float q = m + P2;
                    // absent labels: c = +inf, so L = +inf
                    const float n0 = c.x + (fminf(fminf(q, v0), fminf(left, v1) + P1) - m);
                    const float n1 = c.y + (fminf(fminf(q, v1), fminf(v0, v2) + P1) - m);
                    const float n2 = c.z + (fminf(fminf(q, v2), fminf(v1, v3) + P1) - m);
                    const float n3 = c.w + (fminf(fminf(q, v3), fminf(v2, right) + P1) - m);
                    if (h0) {
                        const float a0 = det_addend(n0, c.x + P2, mk);
                        const float a1 = h1 ? det_addend(n1, c.y + P2, mk) : 0.f;
                        const float a2 = h2 ? det_addend(n2, c.z + P2, mk) : 0.f;
                        const float a3 = h3 ? det_addend(n3, c.w + P2, mk) : 0.f;
                        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                                     ::"l"(ab + 4ll * mt.y), "f"(a0), "f"(a1), "f"(a2), "f"(a3) : "memory");
                    }
                    v0 = n0;
                    v1 = n1;
                    v2 = n2;
                    v3 = n3;
                    m = warp_min(fminf(fminf(n0, n1), fminf(n2, n3)));
                    k++;
                    if ((k & 31) == 0 && k < len) next_block();
                    if (mt1.x != pw || k >= len) break;
                    mt = mt1;
                    c = c1;
                    c1 = c2;
                    mt1 = mt2;
                }
                // the row back to shared memory for what follows
                __syncwarp();
                if (h0) bufA[j0] = v0;
                if (h1) bufA[j0 + 1] = v1;
                if (h2) bufA[j0 + 2] = v2;
                if (h3) bufA[j0 + 3] = v3;
                __syncwarp();
                prev = lane < pn ? bufA[lane] : INF;
                continue;
            }
        }
        const int kb = k & ~31;
        const int kbend = min(kb + 32, len);
        // steps of this block that need the general form: invalid or wider than 32 labels
        const int wn = cw >> 16;
        const unsigned bad = __ballot_sync(0xffffffffu, kb + lane < len && (wn == 0 || wn > 32));
        const unsigned ahead = bad & (0xffffffffu << (k - kb));
        int kend = ahead ? kb + __ffs(ahead) - 1 : kbend;
        if (pn > 32) kend = k;                 // a wide predecessor: the general form takes this step
        if (k < kend && !lead) {
            // SPLIT: the other warps skip to the next general step, knowing only the last narrow
            // step's window
            const int wl = __shfl_sync(0xffffffffu, cw, kend - 1 - kb);
            plo = wl & 0xffff;
            pn = wl >> 16;
            k = kend;
            in_smem = false;
        }
        if (k < kend) {
            // narrow steps: the predecessor row in registers, cost rows two steps ahead
            int ofs = __shfl_sync(0xffffffffu, co, k - kb);
            const int win = __shfl_sync(0xffffffffu, cw, k - kb);
            int l = win & 0xffff, n = win >> 16;
            float c = lane < n ? __ldg(cost + 4ll * ofs + lane) : 0.f;
            int2 mt1 = meta[(k + 1) & 63];
            float c1 = lane < (mt1.x >> 16) ? __ldg(cost + 4ll * mt1.y + lane) : 0.f;
            for (; k < kend; k++) {
                // the metadata of the step after next (from the ring; past the end of the scanline
                // it is zero: no window) and its cost row (a wide row has more than 32 slots, so its
                // first 32 are in bounds too): cost rows two steps ahead
                const int2 mt2 = meta[(k + 2) & 63];
                float c2 = 0.f;
                if (lane < (mt2.x >> 16)) c2 = __ldg(cost + 4ll * mt2.y + lane);
                const int win1 = mt1.x, ofs1 = mt1.y;
                const int n1 = win1 >> 16;
                float Lv = c;
                unsigned cd = 4;
                if (pn != 0) {
                    const int s0 = lane + (l - plo);     // slot of this label in the predecessor
                    const float v0 = __shfl_sync(0xffffffffu, prev, s0 & 31);
                    const float vm = __shfl_sync(0xffffffffu, prev, (s0 - 1) & 31);
                    const float vp = __shfl_sync(0xffffffffu, prev, (s0 + 1) & 31);
                    // min(L'(g-1) + P1, L'(g+1) + P1) = min(L'(g-1), L'(g+1)) + P1 exactly (rounding
                    // is monotone); an absent neighbour is +inf
                    const float a = (unsigned)(s0 - 1) < (unsigned)pn ? vm : INF;
                    const float b = (unsigned)(s0 + 1) < (unsigned)pn ? vp : INF;
                    const float v = (unsigned)s0 < (unsigned)pn ? v0 : INF;
                    float t = fminf(m + P2, fminf(a, b) + P1);
                    t = fminf(t, v);
                    if (REC) cd = t == m + P2 ? 3u : (t == v ? 0u : (t == a + P1 ? 1u : 2u));
                    Lv = c + (t - m);
                }
                const bool act = lane < n;
                if (act) atomicAdd(agg + 4ll * ofs + lane, det_addend(Lv, c + P2, mk));
                prev = act ? Lv : INF;
                m = warp_min(prev);
                if (REC) {
                    if (act) code[4ll * ofs + lane] = (unsigned char)cd;
                    const int slot = (int)__reduce_min_sync(0xffffffffu, prev == m ? (unsigned)lane : 0x7fffffffu);
                    if (lane == 0) am[p0 + (long long)k * dpix] = slot;
                }
                plo = l;
                pn = n;
                l = win1 & 0xffff;
                n = n1;
                ofs = ofs1;
                c = c1;
                c1 = c2;
                mt1 = mt2;
            }
            in_smem = false;
        }
        if (k < kbend) {
            // one general step: an invalid window restarts the path; a window wider than 32 labels
            // (this one or the predecessor's) works on rows by slot in shared memory
            const int win = __shfl_sync(0xffffffffu, cw, k - kb), ofs = __shfl_sync(0xffffffffu, co, k - kb);
            const int l = win & 0xffff, n = win >> 16;
            if (n == 0) {
                pn = 0;
            } else {
                if (pn != 0 && !in_smem) {
                    // the narrow steps' last row (and, SPLIT, its minimum) to shared memory
                    if (lead) {
                        if (lane < pn) bufA[lane] = prev;
                        if (lane == 0) {
                            bufA[pn] = INF;
                            if (SPLIT) xm[4 * NW] = m;
                        }
                    }
                    if (SPLIT) {
                        __syncthreads();
                        m = xm[4 * NW];
                    } else {
                        __syncwarp();
                    }
                }
                const long long o = 4ll * ofs;
                float lmin = INF;
                int lslot = 0x7fffffff;
                if constexpr (SPLIT) {
                    // four consecutive labels a thread; the first vectors of the wide steps up to
                    // kSplitRing - 1 ahead are on their way to the thread's place in the cost rows
                    const int t0 = 4 * (32 * wib + lane);
                    if (asked < k) asked = k;
                    for (; asked < k + kSplitRing; asked++) {
                        const int2 w = meta[asked & 63];
                        if ((w.x >> 16) > 32 && t0 < (w.x >> 16))
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                         ::"r"((unsigned)__cvta_generic_to_shared(cring + (asked & (kSplitRing - 1)) * cstride + t0)),
                                         "l"(cost + 4ll * w.y + t0) : "memory");
                        asm volatile("cp.async.commit_group;" ::: "memory");
                    }
                    asm volatile("cp.async.wait_group %0;" ::"n"(kSplitRing - 1) : "memory");
                    const bool same = l == plo && n == pn;
                    const unsigned top = (unsigned)pn + 1u;
                    for (int j0 = t0; j0 < n; j0 += 128 * NW) {
                        const float4 c4 = j0 == t0 && n > 32
                                              ? *reinterpret_cast<const float4 *>(cring + (k & (kSplitRing - 1)) * cstride + t0)
                                              : __ldg(reinterpret_cast<const float4 *>(cost + o + j0));
                        wide_cells<REC>(c4, j0, n, l, plo, pn, same, top, bufA, m, P1, P2, mk, agg + o,
                                        REC ? code + o : nullptr, lmin, lslot, bufB);
                    }
                }
                // one warp: four vectors of four labels a lane per round, their cost loads in flight together
                // (512^2 pixels, windows of 401 labels at 10 % and 30 % of them: 282 and 503 us, with a label a lane
                // 303 and 565)
                if constexpr (!SPLIT && !REC) {
                    const bool same = l == plo && n == pn;
                    const unsigned top = (unsigned)pn + 1u;
                    for (int jr = 4 * lane; jr < n; jr += 512) {
                        float4 c4[4];
#pragma unroll
                        for (int u = 0; u < 4; u++)
                            c4[u] = jr + 128 * u < n ? __ldg(reinterpret_cast<const float4 *>(cost + o + jr + 128 * u))
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            if (jr + 128 * u >= n) break;
                            wide_cells<REC>(c4[u], jr + 128 * u, n, l, plo, pn, same, top, bufA, m, P1, P2, mk, agg + o,
                                            REC ? code + o : nullptr, lmin, lslot, bufB);
                        }
                    }
                }
                // sixteen of this warp's 32-label chunks per round: their cost loads are in flight
                // together, and every chunk reads the predecessor row before any chunk stores its own
                // (the compiler cannot tell bufA from bufB, so a store between them would order the
                // chunks one after another)
                constexpr int CS = 32;                 // slot stride between the chunks
                if constexpr (REC && !SPLIT)
                for (int j0 = lane; j0 < n; j0 += 16 * CS) {
                    float cc[16];
#pragma unroll
                    for (int u = 0; u < 16; u++) cc[u] = j0 + CS * u < n ? __ldg(cost + o + j0 + CS * u) : 0.f;
                    if (pn != 0) {
                        // predecessor slot s read at row[s + 1] with s + 1 clamped (unsigned) to
                        // pn + 1: any slot outside [0, pn) lands on a sentinel (+inf), so an absent
                        // label drops out of the minimum (labels j >= n read in-bounds slots too)
                        const unsigned top = (unsigned)pn + 1u;
                        const float *row = bufA - 1;
                        auto step = [&](int u, float v0, float vm, float vp) {
                            const float t = fminf(fminf(m + P2, v0), fminf(vm, vp) + P1);
                            code[o + j0 + CS * u] = t == m + P2 ? 3 : (t == v0 ? 0 : (t == vm + P1 ? 1 : 2));
                            const float Ln = cc[u] + (t - m);
                            // the cell's cost cc[u] bounds its path costs (the global atomic does
                            // not order the shared-memory reads of the other chunks)
                            atomicAdd(agg + o + j0 + CS * u, det_addend(Ln, cc[u] + P2, mk));
                            cc[u] = Ln;
                        };
                        if (l == plo && n == pn) {
                            // the same window as the predecessor (a run of whole-range windows):
                            // slot j's neighbours are slots j - 1 and j + 1, and the sentinels at
                            // slots -1 and pn stand in for the absent ones
                            const float *q = bufA + j0;
#pragma unroll
                            for (int u = 0; u < 16; u++) {
                                if (j0 + CS * u >= n) break;
                                step(u, q[CS * u], q[CS * u - 1], q[CS * u + 1]);
                            }
                        } else {
#pragma unroll
                            for (int u = 0; u < 16; u++) {
                                if (j0 + CS * u >= n) break;
                                const unsigned k1 = (unsigned)(l + j0 + CS * u - plo + 1);
                                step(u, row[min(k1, top)], row[min(k1 - 1u, top)], row[min(k1 + 1u, top)]);
                            }
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < 16; u++) {
                            if (j0 + CS * u >= n) break;
                            atomicAdd(agg + o + j0 + CS * u, det_addend(cc[u], cc[u] + P2, mk));
                            code[o + j0 + CS * u] = 4;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 16; u++) {
                        const int j = j0 + CS * u;
                        if (j >= n) break;
                        bufB[j] = cc[u];
                        if (cc[u] < lmin) lslot = j;      // a lane's slots ascend: its first minimum
                        lmin = fminf(lmin, cc[u]);
                    }
                }
                if (SPLIT) {
                    // the warps' minima (and lowest minimising slots) through xm, then the minimum
                    const float wm = warp_min(lmin);
                    int ws = 0;
                    if (REC) ws = (int)__reduce_min_sync(0xffffffffu, lmin == wm ? (unsigned)lslot : 0x7fffffffu);
                    if (lane == 0) {
                        xm[gpar * NW + wib] = wm;
                        if (REC) reinterpret_cast<int *>(xm)[2 * NW + gpar * NW + wib] = ws;
                        if (wib == 0) bufB[n] = INF;
                    }
                    __syncthreads();
                    const float mv = lane < NW ? xm[gpar * NW + lane] : INF;
                    m = warp_min(mv);
                    if (REC) {
                        const unsigned sv = lane < NW && mv == m
                                                ? (unsigned)reinterpret_cast<const int *>(xm)[2 * NW + gpar * NW + lane]
                                                : 0x7fffffffu;
                        const int slot = (int)__reduce_min_sync(0xffffffffu, sv);
                        if (wib == 0 && lane == 0) am[p0 + (long long)k * dpix] = slot;
                    }
                    gpar ^= 1;
                } else {
                    m = warp_min(lmin);
                    if (REC) {
                        const int slot = (int)__reduce_min_sync(0xffffffffu, lmin == m ? (unsigned)lslot : 0x7fffffffu);
                        if (lane == 0) am[p0 + (long long)k * dpix] = slot;
                    }
                    if (lane == 0) bufB[n] = INF;
                    __syncwarp();
                }
                float *tmp = bufA;
                bufA = bufB;
                bufB = tmp;
                if (lead) prev = lane < n ? bufA[lane] : INF;   // for a following narrow step
                in_smem = true;
                plo = l;
                pn = n;
                __syncwarp();
            }
            k++;
        }
        if ((k & 31) == 0 && k < len) next_block();
    }
}

// Two scanlines per warp, sixteen lanes each (half h = lane >> 4), in step: lane i of a half owns slots
// 2i and 2i + 1 of its window (vector loads and reductions).  A narrow step takes about 100 instructions
// for both scanlines instead of 72 for each.  A block of 32 steps is looked over once: the steps that are
// not narrow in both halves (a path start, a window or predecessor wider than 32 labels, an invalid
// window) are taken one by one, and those at which neither window moves need no alignment.
// Wide steps run on the whole warp, first the one half's, then the other's, on rows by slot in shared
// memory (row: the warp's three rows of rstride floats, the halves' and a spare one; slot -1 and slot n hold
// +inf).
// mt: the halves' metadata rings, 64 steps each (as in sgm_scanline).
__device__ __forceinline__ void sgm_pair(const float *__restrict__ cost, const int *__restrict__ lo,
                                         const int *__restrict__ cnt, const long long *__restrict__ off, int H, int W,
                                         float P1, float P2, int G, float *__restrict__ agg, int *__restrict__ status,
                                         int rs, bool have, int mk, float *row, int rstride, int2 *ring) {
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31, i = lane & 15, h = lane >> 4;
    const float INF = __int_as_float(0x7f800000);
    const int r = rs & 15;
    int dx, dy, x0, y0;
    dir_of(r, dx, dy);
    scan_start_d(dx, dy, rs >> 4, H, W, x0, y0);
    const int len = have ? scan_steps(x0, y0, dx, dy, H, W) : 0;
    const int p0 = y0 * W + x0, dpix = dy * W + dx;
    const int maxlen = max(__shfl_sync(ALL, len, 0), __shfl_sync(ALL, len, 16));
    int2 *mt = ring + 64 * h;
    if (lane < 3) row[lane * rstride - 1] = INF;
    // the window metadata of steps kb .. kb + 31 into the half's ring (see sgm_scanline)
    auto fetch = [&](int kb) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = kb + 16 * u + i;
            int2 v = make_int2(0, 0);
            if (k < len) {
                const int p = p0 + k * dpix;
                const int l_ = __ldg(lo + p), n_ = __ldg(cnt + p);
                const long long o_ = __ldg(off + p), e_ = __ldg(off + p + 1);
                if (window_ok(l_, n_, G, e_ - o_, status) && ((o_ | e_) & 3) == 0 && (o_ >> 2) < 0x7fffffff)
                    v = make_int2(l_ | (n_ << 16), (int)(o_ >> 2));
                else if (((o_ | e_) & 3) != 0 && status)
                    atomicExch(status, 7);
            }
            mt[k & 63] = v;
        }
    };
    fetch(0);
    __syncwarp();
    int plo = 0, pn = 0;                          // the half's predecessor window; pn = 0: the path (re)starts
    float v0 = INF, v1 = INF, m = 0.f;            // its slots 2i and 2i + 1 and its minimum
    int in_smem = 0, own = h;                     // its row is (also) in shared memory, in row `own`
    int spare = 2;                                // the row that neither half uses
    const float2 none = make_float2(0.f, 0.f);
    const float *cbase = cost + 2 * i;
    float *abase = agg + 2 * i;
    auto cost_of = [&](int2 w) {
        return 2 * i < (w.x >> 16) ? __ldg(reinterpret_cast<const float2 *>(cbase + 4ll * w.y)) : none;
    };
    // slots s - 1 .. s + 2 of the predecessor row for s = 2i + d, +inf outside [0, 32) (and from pn on)
    auto shifted = [&](int d, float &a, float &b, float &c, float &e) {
        const int q = i + (d >> 1), odd = d & 1, s = 2 * i + d;
        const float B = __shfl_sync(ALL, v0, q, 16), C = __shfl_sync(ALL, v1, q, 16);
        const float D = __shfl_sync(ALL, v0, q + 1, 16), X = __shfl_sync(ALL, v1, q - 1 + 2 * odd, 16);
        a = (unsigned)(s - 1) < 32u ? (odd ? B : X) : INF;
        b = (unsigned)s < 32u ? (odd ? C : B) : INF;
        c = (unsigned)(s + 1) < 32u ? (odd ? D : C) : INF;
        e = (unsigned)(s + 2) < 32u ? (odd ? X : D) : INF;
    };
    // the step on the neighbours a (slot - 1), b, c (the two slots) and e; writes the cells of halves with
    // `on`; returns the new row
    auto cells = [&](float2 cs, int n, int ofs, float a, float b, float c, float e, bool start, bool on, float &n0,
                     float &n1) {
        const float q = m + P2;
        const float t0 = fminf(fminf(q, fminf(a, c) + P1), b), t1 = fminf(fminf(q, fminf(b, e) + P1), c);
        float L0 = cs.x + (t0 - m), L1 = cs.y + (t1 - m);
        if (start) {
            L0 = cs.x;
            L1 = cs.y;
        }
        const bool h0 = on && 2 * i < n, h1 = on && 2 * i + 1 < n;
        if (h0) {
            const float s0 = det_addend(L0, cs.x + P2, mk), s1 = h1 ? det_addend(L1, cs.y + P2, mk) : 0.f;
            asm volatile("red.global.add.v2.f32 [%0], {%1, %2};"
                         ::"l"(abase + 4ll * ofs), "f"(s0), "f"(s1) : "memory");
        }
        n0 = h0 ? L0 : INF;
        n1 = h1 ? L1 : INF;
    };
    auto half_min = [&](float x) {
        const float ma = warp_min(h ? INF : x), mb = warp_min(h ? x : INF);
        return h ? mb : ma;
    };
    for (int kb = 0; kb < maxlen; kb += 32) {
        const int kbend = min(kb + 32, maxlen);
        // the block's steps that are not narrow in both halves, and those at which neither window moves
        unsigned special = 0u, still = 0u;
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int k = kb + 16 * u + i;
            const int w = mt[k & 63].x, pw = k > 0 ? mt[(k - 1) & 63].x : 0;
            const int n = w >> 16, q = pw >> 16;
            const unsigned sp = __ballot_sync(ALL, k < len && ((unsigned)(n - 1) >= 32u || (unsigned)(q - 1) >= 32u));
            const unsigned mv = __ballot_sync(ALL, k < len && (w & 0xffff) != (pw & 0xffff));
            special |= ((sp | sp >> 16) & 0xffffu) << (16 * u);
            still |= (~(mv | mv >> 16) & 0xffffu) << (16 * u);
        }
        __syncwarp();                             // step kb - 1 is read; the next block takes its slots
        fetch(kb + 32);
        __syncwarp();
        int k = kb;
        while (k < kbend) {
            const unsigned ahead = special >> (k - kb);
            const int kend = ahead ? k + __ffs(ahead) - 1 : kbend;
            if (k < kend) {
                // a step on (w, c); (wn, cn) take the metadata and cost row of two steps ahead.  Three register
                // sets in turn, and the cells in both branches: rotating one set took 20 moves a step.
                auto step = [&](const int2 w, const float2 c, int2 &wn, float2 &cn) {
                    wn = mt[(k + 2) & 63];
                    cn = cost_of(wn);
                    const int l = w.x & 0xffff, n = w.x >> 16;
                    if (still >> (k - kb) & 1u) {
                        float a = __shfl_up_sync(ALL, v1, 1, 16), e = __shfl_down_sync(ALL, v0, 1, 16);
                        a = i == 0 ? INF : a;
                        e = i == 15 ? INF : e;
                        cells(c, n, w.y, a, v0, v1, e, false, true, v0, v1);
                    } else {
                        float a, b, cc, e;
                        shifted(l - plo, a, b, cc, e);
                        cells(c, n, w.y, a, b, cc, e, false, true, v0, v1);
                        plo = l;
                    }
                    m = half_min(fminf(v0, v1));
                    return ++k == kend;
                };
                int2 wa = mt[k & 63], wb = mt[(k + 1) & 63], wc;
                float2 ca = cost_of(wa), cb = cost_of(wb), cc;
                for (;;) {
                    if (step(wa, ca, wc, cc)) break;
                    if (step(wb, cb, wa, ca)) break;
                    if (step(wc, cc, wb, cb)) break;
                }
                plo = mt[(k - 1) & 63].x & 0xffff;
                pn = mt[(k - 1) & 63].x >> 16;
                in_smem = 0;
            }
            if (k >= kbend) break;
            // a step that is not narrow in both halves: the half that is, if one is, first
            const int2 w = mt[k & 63];
            const int l = w.x & 0xffff, n = w.x >> 16;
            const bool gen = k < len && (n == 0 || n > 32 || pn > 32), nar = k < len && !gen;
            {
                float a, b, c, e, n0, n1;
                shifted(l - plo, a, b, c, e);
                cells(nar ? cost_of(w) : none, n, w.y, a, b, c, e, pn == 0, nar, n0, n1);
                const float mn = half_min(fminf(n0, n1));
                if (nar) {
                    v0 = n0;
                    v1 = n1;
                    m = mn;
                    plo = l;
                    pn = n;
                    in_smem = 0;
                }
            }
#pragma unroll 1
            for (int hh = 0; hh < 2; hh++) {
                const int src = 16 * hh;
                if (!__shfl_sync(ALL, (int)gen, src)) continue;
                const int gn = __shfl_sync(ALL, n, src), gl = __shfl_sync(ALL, l, src);
                if (gn == 0) {
                    if (h == hh) pn = 0;
                    continue;
                }
                const int gpn = __shfl_sync(ALL, pn, src), gpl = __shfl_sync(ALL, plo, src);
                const int ga = __shfl_sync(ALL, own, src);
                const float gm = __shfl_sync(ALL, m, src);
                const long long o = 4ll * __shfl_sync(ALL, w.y, src);
                float *A = row + ga * rstride, *B = row + spare * rstride;
                if (h == hh && pn != 0 && !in_smem) {      // the narrow steps' last row
                    if (2 * i < pn) A[2 * i] = v0;
                    if (2 * i + 1 < pn) A[2 * i + 1] = v1;
                    if (i == 0) A[pn] = INF;
                }
                __syncwarp();
                float lmin = INF;
                int lslot = 0x7fffffff;
                const bool same = gl == gpl && gn == gpn;
                const unsigned top = (unsigned)gpn + 1u;
                for (int jr = 4 * lane; jr < gn; jr += 256) {
                    float4 c4[2];                          // two vectors' loads in flight together
#pragma unroll
                    for (int u = 0; u < 2; u++)
                        c4[u] = jr + 128 * u < gn ? __ldg(reinterpret_cast<const float4 *>(cost + o + jr + 128 * u))
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int u = 0; u < 2; u++)
                        if (jr + 128 * u < gn)
                            wide_cells<false>(c4[u], jr + 128 * u, gn, gl, gpl, gpn, same, top, A, gm, P1, P2, mk, agg + o,
                                            nullptr, lmin, lslot, B);
                }
                const float mn = warp_min(lmin);
                if (lane == 0) B[gn] = INF;
                __syncwarp();
                if (h == hh) {
                    m = mn;
                    own = spare;
                    plo = gl;
                    pn = gn;
                    in_smem = 1;
                    v0 = 2 * i < gn ? B[2 * i] : INF;      // for a following narrow step
                    v1 = 2 * i + 1 < gn ? B[2 * i + 1] : INF;
                }
                spare = ga;
                __syncwarp();
            }
            k++;
        }
        __syncwarp();
    }
}

// One warp per scanline, WPC warps per CTA; with split (not null), the first scap CTAs take one
// listed scanline each with all their warps (sgm_scanline SPLIT), and the other warps skip the
// listed ones.  split: [0] scanlines listed, [1 .. scap] the list (rs), then the wide windows of each
// scanline and of the image, then 1 if a scanline crosses four times as many as listed ones must
// (count_wide); more than scap listed, or, where every scanline has its warp and none is that much longer
// than the rest, more than alone: none is split.  PAIR: where the image has at most pair_wide wide windows
// (launch_fine_sgm), a warp takes two scanlines (sgm_pair), and the CTAs past them have nothing to do:
// 512^2 pixels without wide windows 174 -> 141 us, 4x4 x 720 x 1280 with 16 directions and 0.6 % of them
// 1163 -> 800 us; both scanlines wait for the wide steps of either.
// Resident CTAs per SM that the register budget must allow: what the one-warp path reaches on its
// own (72 registers without the record, 96 with it; 8 warps: 80 and 128), so that the split path
// (more registers) does not lower the occupancy of every CTA.
__host__ __device__ constexpr int sgm_min_ctas(bool rec, int wpc) {
    return rec ? (wpc == 2 ? 10 : wpc == 4 ? 5 : 2) : (wpc == 2 ? 14 : wpc == 4 ? 7 : 3);
}

// Floats of the rows of fine_sgm_kernel's CTA: two per warp (PAIR: three), slot 0 on 16-byte boundaries, or what a
// split scanline takes (sgm_scanline).
__host__ __device__ constexpr int row_floats(int wpc, int Gs, bool split, bool pair) {
    const int own = wpc * (pair ? 3 : 2) * (Gs + 8), across = split ? 4 + (2 + kSplitRing) * (Gs + 8) : 0;
    return own > across ? own : across;
}

template <bool REC, int WPC, bool PAIR>
__global__ void __launch_bounds__(32 * WPC, sgm_min_ctas(REC, WPC)) fine_sgm_kernel(const float *__restrict__ cost,
                                                                  const int *__restrict__ lo,
                                                                  const int *__restrict__ cnt,
                                                                  const long long *__restrict__ off,
                                                                  int H, int W, int Gs,
                                                                  const float *__restrict__ pen,
                                                                  int G, ScanTable st, float *__restrict__ agg,
                                                                  int *__restrict__ status,
                                                                  const int *__restrict__ order, int mk,
                                                                  unsigned char *__restrict__ codes,
                                                                  int *__restrict__ amin, size_t nnz_cap,
                                                                  const int *__restrict__ split, int scap,
                                                                  int min_wide, int alone, int pair_wide) {
    extern __shared__ __align__(16) float sm[];
    const int wib = threadIdx.x >> 5;
    // rows by slot with one sentinel slot on each side (slot -1 and slot n hold +inf), Gs + 8 floats,
    // two per warp; then per warp a ring of the metadata of this block of 32 steps and the next one,
    // by step mod 64 (read by the narrow steps with one broadcast load); then xm (SPLIT)
    const int rows = row_floats(WPC, Gs, split != nullptr, PAIR);
    int2 *ring = reinterpret_cast<int2 *>(sm + rows), *meta = ring + wib * 64;
    float *xm = sm + rows + (PAIR ? 2 : 1) * WPC * 128;
    const float P1 = __ldg(pen), P2 = __ldg(pen + 1);
    const int total = st.paths == 8 ? st.cum[8] : st.cum[16];   // (no run-time index, see scan_base)
    const int nsplit = split ? __ldg(split) : 0;
    const bool paired = PAIR && __ldg(split + 1 + scap + total) <= pair_wide;
    const bool on = split && (nsplit <= (paired ? scap : alone) || (nsplit <= scap && __ldg(split + 2 + scap + total) != 0));
    if ((int)blockIdx.x < scap) {
        if (!on || (int)blockIdx.x >= nsplit) return;
        float *bufA = sm + 4;                   // the split rows on 16-byte boundaries, Gs + 8 floats
        sgm_scanline<REC, true, WPC>(cost, lo, cnt, off, H, W, P1, P2, G, agg, status, __ldg(split + 1 + blockIdx.x),
                                     mk, codes, amin, nnz_cap, bufA, bufA + (Gs + 8), meta, xm, wib,
                                     bufA + 2 * (Gs + 8), Gs + 8);
        return;
    }
    const int gw = ((int)blockIdx.x - scap) * WPC + wib;
    if constexpr (PAIR) {
        if (paired) {
            if (2 * gw >= total) return;
            const int q = 2 * gw + ((threadIdx.x >> 4) & 1);
            const int rs = q < total ? __ldg(order + q) : 0;
            const bool have = q < total && !(on && __ldg(split + 1 + scap + scan_base(st, rs & 15) + (rs >> 4)) >= min_wide);
            sgm_pair(cost, lo, cnt, off, H, W, P1, P2, G, agg, status, rs, have, mk,
                     sm + (size_t)wib * 3 * (Gs + 8) + 4, Gs + 8, ring + 128 * wib);
            return;
        }
    }
    if (gw >= total) return;
    const int rs = __ldg(order + gw);            // longest scanlines first
    if (on && __ldg(split + 1 + scap + scan_base(st, rs & 15) + (rs >> 4)) >= min_wide) return;
    float *bufA = sm + (size_t)wib * 2 * (Gs + 8) + 4;
    sgm_scanline<REC, false, 1>(cost, lo, cnt, off, H, W, P1, P2, G, agg, status, rs, mk, codes, amin, nnz_cap,
                                bufA, bufA + (Gs + 8), meta, xm, wib);
}

// The scanlines to split: every pixel with a window wider than 32 labels counts on its scanline of each
// direction (tab[1 + kSplitCap + id]); the one that reaches min_wide lists the scanline (tab[0] listed,
// tab[1 .. kSplitCap] the list, up to kSplitCap of them: the list's order does not matter, every
// scanline's values are its own).  Table zeroed before.  Such pixels are few where splitting pays, so
// this costs the kernels that walk the windows anyway (mean cost, clearing the aggregate) no time; a
// warp per scanline that counts them took 10 us for 8 directions of 512^2, 15 for 16 of 720 x 1280.
// Called by a warp, lane i with pixel p0 + i, wide: its pixels with such windows; the lanes take
// (pixel, direction) pairs, so that a few pixels wait for one round of atomics.
__device__ __forceinline__ void count_wide(unsigned wide, int p0, int W, int H, const ScanTable &st, int min_wide,
                                           int *tab) {
    if (wide == 0u) return;
    const int lane = threadIdx.x & 31, items = __popc(wide) * st.paths;
    if (lane == 0) atomicAdd(tab + 1 + kSplitCap + st.cum[st.paths], __popc(wide));
    if (__ldcg(tab) > kSplitCap) return;                   // too many listed: none is split
    for (int i = lane; i < items; i += 32) {
        const int k = st.paths == 8 ? i >> 3 : i >> 4, r = i - k * st.paths;
        const int p = p0 + (int)__fns(wide, 0, k + 1);
        const int y = p / W, x = p - y * W;
        int dx, dy;
        dir_of(r, dx, dy);
        const int base = scan_base(st, r);
        const int q = scan_index_d(dx, dy, x, y, H, W);
        const int before = atomicAdd(tab + 1 + kSplitCap + base + q, 1);
        if (before == 4 * min_wide - 1) tab[2 + kSplitCap + st.cum[st.paths]] = 1;
        if (before == min_wide - 1) {
            const int pos = atomicAdd(tab, 1);
            if (pos < kSplitCap) tab[1 + pos] = (q << 4) | r;
        }
    }
}

// The aggregate's rows to zero; with tab, the scanlines to split (count_wide).
__global__ void __launch_bounds__(256) zero_agg_kernel(float *__restrict__ agg, const int *__restrict__ cnt,
                                                       const long long *__restrict__ off, int N, int W, int H,
                                                       ScanTable st, int min_wide, int *__restrict__ tab) {
    const long long n = off[N], i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (tab)
        for (long long p = i0; p - (threadIdx.x & 31) < N; p += stride)
            count_wide(__ballot_sync(0xffffffffu, p < N && __ldg(cnt + p) > 32), (int)p - (threadIdx.x & 31), W, H, st,
                       min_wide, tab);
    zero_rows(agg, n, i0, stride);
}

// Per-block sums of the active costs and slot counts (rows are 16-byte aligned, read as float4;
// slots past cnt are masked, so padding is never read into the sum).  The warps take 32
// consecutive pixels at a time, a lane its pixel: a lane sums its row's first 32 slots (8 vector
// loads issued together), and the slots past 32 of a few wide rows in the warp are then summed by
// the whole warp, one row after another (a lane a vector, the lanes' parts added in a fixed
// order), so that one wide row does not hold its warp for a dependent load per 32 slots.  Each
// lane adds its pixels in a fixed order, the block adds its warps in a fixed order, and the last
// block to finish (ticket counter) adds the block partials in block order and writes the
// penalties: the mean is deterministic.  The first nb blocks do this and, with tab, list the SGM
// scanlines to split (count_wide); the blocks past them set the aggregate's rows to 0, beside sums
// that wait for memory (9x9 x 512^2: 33 + 10 us as two kernels, 36 in one).
__global__ void __launch_bounds__(256) cost_partial_kernel(const float *__restrict__ cost,
                                                           const int *__restrict__ cnt,
                                                           const long long *__restrict__ off, int N, int G,
                                                           double *__restrict__ partial, int nb, double p1f,
                                                           double p2f, float *__restrict__ pen,
                                                           unsigned *__restrict__ ticket, int *__restrict__ status,
                                                           int H, int W, ScanTable st, int min_wide,
                                                           int *__restrict__ tab, float *__restrict__ agg) {
    if ((int)blockIdx.x >= nb) {
        zero_rows(agg, off[N], (long long)((int)blockIdx.x - nb) * blockDim.x + threadIdx.x,
                  (long long)((int)gridDim.x - nb) * blockDim.x);
        return;
    }
    double s = 0.0, c = 0.0;
    const int lane0 = threadIdx.x & 31;
    const int wstride = nb * blockDim.x;
    for (int base = blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < N; base += wstride) {
        const int p = base + lane0;
        long long o = 0;
        int n = 0;
        if (p < N) {
            o = off[p];
            n = cnt[p];
            if (!window_ok(0, n, G, off[p + 1] - o, status) || !row_aligned(o, status) ||
                !row_aligned(off[p + 1], status))
                n = 0;
        }
        const float4 *r = reinterpret_cast<const float4 *>(cost + o);
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; q++) v[q] = 4 * q < n ? __ldg(r + q) : make_float4(0.f, 0.f, 0.f, 0.f);
        float ps = 0.f;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int j = 4 * q;
            ps += (j < n ? v[q].x : 0.f) + (j + 1 < n ? v[q].y : 0.f) + (j + 2 < n ? v[q].z : 0.f) +
                  (j + 3 < n ? v[q].w : 0.f);
        }
        // the slots past 32 of this warp's wide rows: a few are summed by the whole warp, one row at
        // a time; when most rows are wide (whole-range searches) each lane sums its own in 32-slot
        // chunks of 8 vector loads issued together
        unsigned wide = __ballot_sync(0xffffffffu, n > 32);
        if (tab) count_wide(wide, base, W, H, st, min_wide, tab);
        if (__popc(wide) > 4) {
            for (int j0 = 32; j0 < n; j0 += 32) {
#pragma unroll
                for (int q = 0; q < 8; q++)
                    v[q] = j0 + 4 * q < n ? __ldg(r + (j0 >> 2) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const int j = j0 + 4 * q;
                    if (j < n)
                        ps += v[q].x + (j + 1 < n ? v[q].y : 0.f) + (j + 2 < n ? v[q].z : 0.f) +
                              (j + 3 < n ? v[q].w : 0.f);
                }
            }
            wide = 0u;
        }
        while (wide) {
            const int src = __ffs(wide) - 1;
            wide &= wide - 1;
            const long long ow = __shfl_sync(0xffffffffu, o, src);
            const int nw = __shfl_sync(0xffffffffu, n, src);
            const float4 *rw = reinterpret_cast<const float4 *>(cost + ow);
            float t = 0.f;
            for (int j = 32 + 4 * lane0; j < nw; j += 128) {
                const float4 a = __ldg(rw + (j >> 2));
                t += a.x + (j + 1 < nw ? a.y : 0.f) + (j + 2 < nw ? a.z : 0.f) + (j + 3 < nw ? a.w : 0.f);
            }
#pragma unroll
            for (int k = 16; k > 0; k >>= 1) t += __shfl_xor_sync(0xffffffffu, t, k);
            if (lane0 == src) ps += t;
        }
        s += (double)ps;
        c += n;
    }
    for (int k = 16; k > 0; k >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, k);
        c += __shfl_down_sync(0xffffffffu, c, k);
    }
    __shared__ double ws[32], wc[32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        ws[wid] = s;
        wc[wid] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0, bc = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) {
            b += ws[i];
            bc += wc[i];
        }
        partial[blockIdx.x] = b;
        partial[nb + blockIdx.x] = bc;
        __threadfence();                                   // partials visible before the ticket
        last = atomicAdd(ticket, 1u) == (unsigned)nb - 1;
    }
    __syncthreads();
    if (!last || wid != 0) return;
    // the last block: all partials are written; add them in block order (a lane every 32nd, eight
    // of them loaded together: one L2 round trip per 256 partials instead of one per 32)
    s = 0.0;
    c = 0.0;
    for (int i0 = lane; i0 < nb; i0 += 256) {
        double sv[8], cv[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int i = i0 + 32 * u;
            sv[u] = i < nb ? __ldcg(partial + i) : 0.0;
            cv[u] = i < nb ? __ldcg(partial + nb + i) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; u++) {
            s += sv[u];
            c += cv[u];
        }
    }
    for (int k = 16; k > 0; k >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, k);
        c += __shfl_down_sync(0xffffffffu, c, k);
    }
    if (lane == 0) {
        const double mean = c > 0.0 ? s / c : 0.0;
        pen[0] = (float)(p1f * mean);
        pen[1] = (float)(p2f * mean);
        *ticket = 0u;                                      // ready for the next launch
    }
}

}  // namespace

cudaError_t launch_cost_partial_sums(cudaStream_t s, const float *cost, const int *cnt, const long long *off,
                                     int N, int G, double *partial, int nblocks, double p1f, double p2f,
                                     float *pen, unsigned *ticket, int *status, int H, int W, int paths,
                                     int min_wide, int *tab, float *agg) {
    // zeroing: a thread per 8 vectors of rows of about 32 slots, four CTAs per SM at most
    const int zero = std::max(1, std::min(608, N / 256));
    cost_partial_kernel<<<nblocks + zero, 256, 0, s>>>(cost, cnt, off, N, G, partial, nblocks, p1f, p2f, pen, ticket,
                                                       status, H, W, make_scan_table(H, W, paths), min_wide, tab, agg);
    return cudaGetLastError();
}
cudaError_t launch_zero_agg(cudaStream_t s, float *agg, const int *cnt, const long long *off, int H, int W, int paths,
                            int min_wide, int *tab) {
    zero_agg_kernel<<<1216, 256, 0, s>>>(agg, cnt, off, H * W, W, H, make_scan_table(H, W, paths), min_wide, tab);
    return cudaGetLastError();
}

void build_scan_order(int H, int W, int paths, std::vector<int> &order) {
    order.clear();
    for (int r = 0; r < paths; r++)
        for (int s = 0; s < n_scanlines(r, H, W); s++) order.push_back((s << 4) | r);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return scan_len(a & 15, a >> 4, H, W) > scan_len(b & 15, b >> 4, H, W);
    });
}

int sgm_split_ints(int H, int W, int paths) {
    return 1 + kSplitCap + make_scan_table(H, W, paths).cum[paths] + 2;
}

cudaError_t launch_fine_sgm(cudaStream_t s, const float *cost, const int *lo, const int *cnt,
                            const long long *off, int H, int W, int G, const float *pen, float *agg,
                            int *status, const int *order, int paths, unsigned char *codes, int *amin,
                            size_t nnz_cap, int warps_per_cta, int min_wide, const int *split, int alone, bool narrow) {
    const int wpc = warps_per_cta == 2 || warps_per_cta == 8 ? warps_per_cta : kSgmWarps;
    const ScanTable st = make_scan_table(H, W, paths);
    const int Gs = (G + 31) & ~31;
    // two scanlines a warp: windows of at most 32 labels where the initial map holds, enough scanlines to keep
    // the SMs busy, and rows that leave room for as many CTAs as the registers do
    const size_t rest = (size_t)(4 * wpc + 4) * 4;
    const size_t psmem = row_floats(wpc, Gs, split, true) * sizeof(float) + (size_t)wpc * 128 * sizeof(int2) + rest;
    const bool pair = split && narrow && !codes && st.cum[paths] >= kPairFrom && psmem * 28 <= (size_t)wpc * 224 * 1024;
    const size_t smem =
        pair ? psmem : row_floats(wpc, Gs, split, false) * sizeof(float) + (size_t)wpc * 64 * sizeof(int2) + rest;
    // Wide windows up to which they do: a pair's time is that of its longest scanline, with the wide steps of
    // both, so the line rises with the steps that a place in flight takes, in longest scanlines, and falls with
    // the labels of a wide step.  One scanline a warp and two, us: 512^2, 8 directions, 401 labels, 0.9 %: 188, 181,
    // 1.6 %: 197, 218; 121 labels, 2 %: 191, 171, 5.6 %: 183, 231; 512^2, 16 directions, 401 labels, 3.4 %: 381, 340,
    // 5.6 %: 436, 450; 300^2, 8 directions, 201 labels, 0.9 %: 85, 88; 720 x 1280, 16 directions, 241 labels, 2 %: 1232,
    // 817, 5.8 %: 1425, 1007.  (A line at 1 % whatever the shape left the last two at 1232 and 1425.)
    const double steps = (double)paths * H * W / kPairPlaces / std::max(H, W);
    const int pair_wide = (int)(std::min(1.0, std::max(0.5, 20.0 * (steps - 0.31)) / G) * H * W);
    const int scap = split ? kSplitCap : 0;
    const unsigned grid = (unsigned)(scap + (st.cum[paths] + wpc - 1) / wpc);
    // one instantiation per CTA size, each with its own register budget (launch bounds)
#define LFSGM_FINE(R, P) (wpc == 2 ? fine_sgm_kernel<R, 2, P> : wpc == 8 ? fine_sgm_kernel<R, 8, P> : fine_sgm_kernel<R, 4, P>)
    auto kern = codes ? LFSGM_FINE(true, false) : pair ? LFSGM_FINE(false, true) : LFSGM_FINE(false, false);
#undef LFSGM_FINE
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int lp = 0;
    while ((1 << lp) < paths) lp++;
    const int mk = (lp << 23) | (1 << 22);       // (23 - qsh) << 23 with qsh = 23 - log2(paths)
    kern<<<grid, 32 * wpc, smem, s>>>(cost, lo, cnt, off, H, W, Gs, pen, G, st, agg, status, order, mk, codes,
                                      amin, nnz_cap, split, scap, min_wide, std::min(alone, scap), pair_wide);
    return cudaGetLastError();
}

}  // namespace lfsgm

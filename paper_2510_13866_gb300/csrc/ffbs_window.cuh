// ffbs_window.cuh -- backward draw of one wide-lattice worldline by one warp from a window
// of f around the worldline (FP32, Hirsch fields).
//
// The backward conditional x_i ~ max(f_i(y), 0) G(x_{i+1} - y) is a row-major inverse CDF over
// all N sites, but G falls off as (t dtau)^d / d!: at t dtau = 0.05 a site ten steps away
// carries G < 2^-65 of the centre.  Reading the whole of f back made the backward pass a
// second stream over HBM of the size of the forward pass's (27% of a sweep at L = 64 and 128,
// 33% with L = 48).  Here a warp reads (2H+1) lines x 28 elements around x_{i+1} (2.7 KB
// instead of 16 KB at L = 64, 64 KB at L = 128) and draws from them alone.
//
// The draw is the same but for 2^-36 of its probability.  Sites beyond WinR steps hold at most
//     g(WinR + 1) g(0) sum_y f(y) <= 4 g(WinR + 1) g(0) max W
// of the conditional's total S (the message is normalised to a sum in [1, 2)); the window
// answers only where that is below 2^-36 S (S >= win_min, a per-chain constant): 4096 times
// below the rounding of S itself and of the 24-bit uniform, though a target near the start of the
// CDF is compared at a finer spacing than that, and such a draw may differ.  Inside the window the
// arithmetic is the whole row's: the same in-row prefix in the order of x, and row totals scanned
// in the association of the whole-slice form (rows outside the window enter as zeros), so all other
// draws are equal.  Where a vanishing weight could still decide -- a uniform of 0, a target equal to
// a row boundary, no crossing -- the warp draws from the whole slice (draw_whole), row by row.
//
// Loads run kWinStages slices ahead, centred on the worldline's site at that time; the margin
// kWinH - WinR covers the steps in between, and a worldline that left it (4 steps one way in
// three slices at t dtau = 0.05: 1e-4 of draws) loads its window again.
#pragma once

#include "device_common.cuh"
#include "internal.h"
#include "window_rule.h"

namespace hqmc {

constexpr int kWinH = kWinHalf;           // lines each side of the centre
constexpr int kWinLines = 2 * kWinH + 1;  // 25
constexpr int kWinChunks = 7;             // aligned 16-byte chunks that hold 2 H + 1 elements at any offset
constexpr int kWinCols = 4 * kWinChunks;
constexpr int kWinStages = 4;
static_assert(kWinLines + 3 <= kWinCols && kWinCols <= 32, "window geometry");
// a stage holds chunk j of line q at 16-byte unit j * kWinLines + q: with 25 lines (1 mod 8) the
// reads of one element of every row (C slices) hit distinct banks
static_assert(kWinLines % 8 == 1, "bank-conflict-free element reads");
constexpr size_t kWinStageBytes = size_t(kWinChunks) * kWinLines * 16;
// per warp: the stages, the x-weights of the window's columns, the crossing row's prefixes
constexpr size_t kWinBytes = kWinStages * kWinStageBytes + 2 * 32 * sizeof(float);

// One window around (cx, cy) of slice i (lines are y in even slices, x in odd ones).  Its chunks
// and lines are kept in the order of their coordinates: what lies past the lattice's edge (nwc
// chunks, nwl lines) comes first, so that the draw's loops run straight through.
template <int L>
struct WinPlace {
    int a0, l0, nwc, nwl;
    __device__ __forceinline__ WinPlace(int i, int cx, int cy) {
        const int ce = (i & 1) ? cy : cx, cl = (i & 1) ? cx : cy;
        const int e0 = ce - kWinH < 0 ? ce - kWinH + L : ce - kWinH;
        a0 = e0 >> 2;
        l0 = cl - kWinH < 0 ? cl - kWinH + L : cl - kWinH;
        nwc = max(0, a0 + kWinChunks - L / 4);
        nwl = max(0, l0 + kWinLines - L);
    }
    // coordinate of element position c, of line position q
    __device__ __forceinline__ int elem(int c) const { return (c >> 2) < nwc ? c : c + 4 * (a0 - nwc); }
    __device__ __forceinline__ int line(int q) const { return q < nwl ? q : q + l0 - nwl; }
};

// asynchronous copy of a window of slice f (one commit group follows)
template <int L>
__device__ __forceinline__ void win_load(unsigned char *stage, const float *f, const WinPlace<L> &w, int lane) {
    if (lane < kWinLines) {
        const float *src = f + w.line(lane) * 4;
        unsigned char *dst = stage + lane * 16;
#pragma unroll
        for (int j = 0; j < kWinChunks; ++j) {
            const int a = j < w.nwc ? j : j + w.a0 - w.nwc;
            cp_async16(dst + j * (kWinLines * 16), src + a * (L * 4));
        }
    }
}

// Draw from the window in `stage` (placed by w); returns row << 8 | column, or -1 where the whole
// slice has to be asked.  `wx`: 32 x-weights, then 32 prefixes (shared memory of the warp).
// SEG: rows that the whole-slice form scans together (the rows of one worldline in a warp).
template <int L, int SEG>
__device__ __forceinline__ int win_draw(const unsigned char *stage, float *wx, const float *g2, int i, const WinPlace<L> &w,
                                        int cx, int cy, uint32_t u24, float smin, int lane) {
    constexpr int NSEG = L / SEG;
    static_assert(SEG == 32 || (SEG == 16 && NSEG == 3), "row segments");
    const bool C = (i & 1) != 0;  // lines are x (else y)
    const int ce = w.elem(lane), cl = w.line(lane);  // of element position and line position `lane`
    const int row = C ? ce : cl, nrow = C ? kWinCols : kWinLines;
    {
        // x-weights of the columns (0 beyond them), y-weight of the row
        const int x = C ? cl : ce, ncol = C ? kWinLines : kWinCols;
        wx[lane] = lane < ncol ? g2[x - cx + L] : 0.f;
    }
    const float gy = lane < nrow ? g2[row - cy + L] : 0.f;
    __syncwarp();
    // inclusive in-row prefix in the order of x
    float pre[kWinCols];
    float P = 0.f;
    const float4 *w4 = reinterpret_cast<const float4 *>(wx);
    if (!C) {
        const float4 *src = reinterpret_cast<const float4 *>(stage) + min(lane, kWinLines - 1);
#pragma unroll
        for (int k = 0; k < kWinChunks; ++k) {
            const float4 f = src[k * kWinLines], q = w4[k];
            P = fmaf(fmaxf(f.x, 0.f), q.x * gy, P);
            pre[4 * k] = P;
            P = fmaf(fmaxf(f.y, 0.f), q.y * gy, P);
            pre[4 * k + 1] = P;
            P = fmaf(fmaxf(f.z, 0.f), q.z * gy, P);
            pre[4 * k + 2] = P;
            P = fmaf(fmaxf(f.w, 0.f), q.w * gy, P);
            pre[4 * k + 3] = P;
        }
    } else {
        const int c = min(lane, kWinCols - 1);
        const float *src = reinterpret_cast<const float *>(stage) + (c >> 2) * (kWinLines * 4) + (c & 3);
#pragma unroll
        for (int k = 0; k < kWinChunks; ++k) {
            const float4 q = w4[k];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (4 * k + e < kWinLines)
                    P = fmaf(fmaxf(src[(4 * k + e) * 4], 0.f), (e == 0 ? q.x : e == 1 ? q.y : e == 2 ? q.z : q.w) * gy, P);
                pre[4 * k + e] = P;
            }
        }
    }
    // Row totals in the association of the whole slice: a scan over the rows of each segment, then
    // the segments in order.  The window touches at most two segments of 32 rows (A before B), or
    // the three of 16: rows 0..31 in vector A, 32..47 in B.
    const int r0 = C ? 4 * w.a0 : w.l0;        // window rows are r0 .. r0 + nrow - 1 (cyclic);
    const int nwr = C ? 4 * w.nwc : w.nwl;     // nwr of them past the edge, at positions 0 ..
    int ra, rb;                                // this lane's row in each vector
    if (SEG == 32) {
        const int s0 = r0 / SEG, s1 = s0 + 1 == NSEG ? 0 : s0 + 1;
        ra = min(s0, s1) * SEG + lane;
        rb = max(s0, s1) * SEG + lane;
    } else {
        ra = lane;
        rb = 32 + (lane & 15);
    }
    // window position of a row, or 32 outside
    auto pos = [&](int r) { return r < nwr ? r : (r >= r0 && r < r0 + nrow) ? r - r0 + nwr : 32; };
    const int wa = pos(ra), wb = pos(rb);
    const float sa = __shfl_sync(0xffffffffu, P, wa), sb = __shfl_sync(0xffffffffu, P, wb);
    const float pa = wa < 32 ? sa : 0.f, pb = wb < 32 ? sb : 0.f;
    float ia = pa, ib = pb;
    const int rs = lane % SEG;
#pragma unroll
    for (int o = 1; o < SEG; o <<= 1) {
        const float ta = __shfl_up_sync(0xffffffffu, ia, o, SEG), tb = __shfl_up_sync(0xffffffffu, ib, o, SEG);
        if (rs >= o) {
            ia += ta;
            ib += tb;
        }
    }
    float xa, xb, S;  // exclusive offsets of the lane's rows in each vector
    const float T0 = __shfl_sync(0xffffffffu, ia, SEG - 1);
    if (SEG == 32) {
        S = T0 + __shfl_sync(0xffffffffu, ib, 31);
        xa = ia - pa;
        xb = T0 + ib - pb;
    } else {
        const float T1 = __shfl_sync(0xffffffffu, ia, 31);
        const float b2 = T0 + T1;
        S = b2 + __shfl_sync(0xffffffffu, ib, 15);
        xa = (lane < 16 ? 0.f : T0) + ia - pa;
        xb = b2 + ib - pb;
    }
    const float t = __fmul_rd(float(u24) * 0x1.0p-24f, S);
    // no answer: a total below win_min (or not a number), a uniform of 0, or a target equal to a row
    // boundary, where an outside row or column of vanishing weight could hold it
    const bool edge = !(S >= smin) || !(S < 1e30f) || u24 == 0u || t == xa || t == xb || t == T0 || t == S;
    // back to the window's rows
    const float ea = __shfl_sync(0xffffffffu, xa, row & 31), eb = __shfl_sync(0xffffffffu, xb, SEG == 32 ? row & 31 : row & 15);
    const float ex = (SEG == 32 ? (row ^ ra) < 32 : row < 32) ? ea : eb;
    const float rem = t - ex;
    // the first row of the lattice whose total exceeds what remains of u S
    const unsigned hit = __ballot_sync(0xffffffffu, lane < nrow && t >= ex && P > rem);
    if (__any_sync(0xffffffffu, edge) || hit == 0u) return -1;
    const int win = __ffs(hit) - 1;
    // and in it the first column whose prefix does
    float *pr = wx + 32;
    if (lane == win) {
#pragma unroll
        for (int k = 0; k < kWinChunks; ++k)
            reinterpret_cast<float4 *>(pr)[k] = make_float4(pre[4 * k], pre[4 * k + 1], pre[4 * k + 2], pre[4 * k + 3]);
    }
    const float wrem = __shfl_sync(0xffffffffu, rem, win);
    __syncwarp();
    const int n = __ffs(__ballot_sync(0xffffffffu, lane < kWinCols && pr[lane] > wrem)) - 1;
    return C ? (w.elem(win) << 8 | w.line(n)) : (w.line(win) << 8 | w.elem(n));
}

// The same draw from the whole slice, by one warp, row by row from memory (rare: a worldline
// in a region where the message has sunk to the FFT's rounding floor).  Returns row << 8 | column,
// or -1 for an all-zero CDF.
template <int L, int SEG>
__device__ __noinline__ int draw_whole(const float *f, const float *g2, int i, int cx, int cy, uint32_t u24, int lane) {
    constexpr int NSEG = L / SEG;
    const bool C = (i & 1) != 0;
    const int rs = lane % SEG;
    auto at = [&](int x, int y) {
        const int line = C ? x : y, e = C ? y : x;
        return fmaxf(__ldcg(f + ((e >> 2) * L + line) * 4 + (e & 3)), 0.f);
    };
    float P[NSEG], ex[NSEG], base = 0.f;
#pragma unroll
    for (int k = 0; k < NSEG; ++k) {
        const int y = k * SEG + rs;
        const float gy = g2[y - cy + L];
        float p = 0.f;
#pragma unroll 32  // loads in flight: this is the latency of memory, L / 32 times per row
        for (int x = 0; x < L; ++x) p = fmaf(at(x, y), g2[x - cx + L] * gy, p);
        float inc = p;
#pragma unroll
        for (int o = 1; o < SEG; o <<= 1) {
            const float t0 = __shfl_up_sync(0xffffffffu, inc, o, SEG);
            if (rs >= o) inc += t0;
        }
        P[k] = p;
        ex[k] = base + inc - p;
        base += __shfl_sync(0xffffffffu, inc, SEG - 1);
    }
    if (!(base > 0.f)) return -1;
    const float t = __fmul_rd(float(u24) * 0x1.0p-24f, base);
    int row = 0x7fffffff;
    float rem = 0.f;
#pragma unroll
    for (int k = NSEG - 1; k >= 0; --k) {
        const float r = t - ex[k];
        if (t >= ex[k] && P[k] > r) {
            row = k * SEG + rs;
            rem = r;
        }
    }
    const int win = __reduce_min_sync(0xffffffffu, row);
    if (win != 0x7fffffff) {
        // the row that holds the crossing, its first column past the remainder
        rem = __shfl_sync(0xffffffffu, rem, __ffs(__ballot_sync(0xffffffffu, row == win)) - 1);
        const float gy = g2[win - cy + L];
        float p = 0.f;
        int n = 0;
#pragma unroll 32
        for (int x = 0; x < L; ++x) {
            p = fmaf(at(x, win), g2[x - cx + L] * gy, p);
            n += (p <= rem) ? 1 : 0;
        }
        return win << 8 | n;
    }
    // u*S at or beyond the rounded total: the last site with a positive weight
    int last = -1;
    for (int k = 0; k < NSEG; ++k) {
        const int y = k * SEG + rs;
        const float gy = g2[y - cy + L];
        float p = 0.f;
        for (int x = 0; x < L; ++x) {
            const float q = fmaf(at(x, y), g2[x - cx + L] * gy, p);
            if (q > p) last = max(last, y << 8 | x);
            p = q;
        }
    }
    return __reduce_max_sync(0xffffffffu, last);
}

// A unit whose forward pass is done and whose worldlines are still to be drawn.
struct WinUnit {
    int c, sg, pw0, nwl;  // chain, spin, first worldline, worldlines present
    int l0, len, le, wi;  // first slice, block length, last slice, first position past the wrap
    int normal[2];        // every stored f of the worldline is normalised
};

// Backward pass of worldline k of a unit by one warp.  f: its slot; g2, hl: the chain's doubled
// ring propagator and link table (shared memory); ring: kWinBytes of the warp's.
template <int L, int WPC>
__device__ __forceinline__ void win_backward(const DevState &st, const WinUnit &un, int k, const float *f, const float *g2,
                                             const float *hl, unsigned char *ring, uint64_t sweep, int lane) {
    constexpr int N = L * L;
    const int c = un.c, sg = un.sg, pk = un.pw0 + k, l0 = un.l0, len = un.len, wi = un.wi;
    const ChainDev &cd = st.chains[c];
    const int M = cd.M, Nsig = cd.Nsig, margin = kWinH - cd.win_R;
    int16_t *xspin = st.x + cd.x_off + (long long)sg * Nsig * M;
    const int qk = st.perm[cd.perm_off + sg * Nsig + pk];
    int16_t *own_p = xspin + (long long)pk * M, *own_q = xspin + (long long)qk * M;
    float *wx = reinterpret_cast<float *>(ring + kWinStages * kWinStageBytes);
    const float smin = un.normal[k] ? cd.win_min : __int_as_float(0x7f800000);
    const uint64_t wl = (uint64_t)sg * Nsig + pk, seed = cd.seed;
    int *hist = st.hist + cd.h_off + (long long)sg * M * N;
    const int xs = (0 >= wi ? own_q : own_p)[l0];
    int cx, cy;
    {
        const int xe = (len >= wi ? own_q : own_p)[un.le];
        cx = xe % L;
        cy = xe / L;
    }
    uint64_t ctr = 0;  // centres of the stages' windows, 16 bits each
    auto load = [&](int i) {
        const int sh = 16 * (i & (kWinStages - 1));
        ctr = (ctr & ~(0xffffull << sh)) | (uint64_t(cx | (cy << 8)) << sh);
        win_load<L>(ring + (i & (kWinStages - 1)) * kWinStageBytes, f + (long long)i * N, WinPlace<L>(i, cx, cy), lane);
    };
    auto wrap = [](int d) { return d < 0 ? d + L : d; };
    if (lane == 0) atomicAdd(hist + (long long)l0 * N + xs, 1);
    float ek = 0.f;
    int cached = -1;
    uint32_t wd0 = 0, wd1 = 0, wd2 = 0, wd3 = 0;  // leading 24 bits of the words
    // the windows of the first positions, then one iteration per slice
#pragma unroll 1
    for (int i = len + kWinStages - 2; i >= 1; --i) {
        __syncwarp();  // the slice that used this stage has been read
        if (i - kWinStages + 1 >= 1) load(i - kWinStages + 1);
        cp_async_commit();
        if (i >= len) continue;
        int lb = l0 + i;
        if (lb >= M) lb -= M;
        // uniforms: lane g keeps the words of group g of 32 groups of four slices
        const int grp = lb >> 2, blk = grp >> 5;
        if (blk != cached) {
            const u64x4 w4 = philox4x64_10((uint64_t)(blk * 32 + lane), wl, 0, sweep, seed, 0);
            wd0 = uint32_t(w4.v[0] >> 40);
            wd1 = uint32_t(w4.v[1] >> 40);
            wd2 = uint32_t(w4.v[2] >> 40);
            wd3 = uint32_t(w4.v[3] >> 40);
            cached = blk;
        }
        const uint32_t u24 = __shfl_sync(
            0xffffffffu, (lb & 2) ? ((lb & 1) ? wd3 : wd2) : ((lb & 1) ? wd1 : wd0), grp & 31);
        cp_async_wait<kWinStages - 1>();
        const uint32_t ct = uint32_t(ctr >> (16 * (i & (kWinStages - 1))));
        int wcx = ct & 0xff, wcy = (ct >> 8) & 0xff;
        const int dx = abs(cx - wcx), dy = abs(cy - wcy);
        if (max(min(dx, L - dx), min(dy, L - dy)) > margin) {
            // the worldline left the window's margin: load it again
            __syncwarp();
            load(i);
            cp_async_commit();
            cp_async_wait_all();
            wcx = cx;
            wcy = cy;
        }
        __syncwarp();
        int nxt = win_draw<L, 32 / WPC>(ring + (i & (kWinStages - 1)) * kWinStageBytes, wx, g2, i, WinPlace<L>(i, wcx, wcy),
                                        cx, cy, u24, smin, lane);
        if (nxt < 0) {
            nxt = draw_whole<L, 32 / WPC>(f + (long long)i * N, g2, i, cx, cy, u24, lane);
            if (nxt < 0) {
                if (lane == 0) atomicAdd(&st.meas[c].degenerate, 1ull);
                nxt = cy << 8 | cx;
            }
        }
        const int nx = nxt & 0xff, ny = nxt >> 8;
        if (lane == 0) {
            ek += hl[wrap(cx - nx)] + hl[wrap(cy - ny)];
            (i >= wi ? own_q : own_p)[lb] = int16_t(nx + L * ny);
            atomicAdd(hist + lb * N + nx + L * ny, 1);
        }
        cx = nx;
        cy = ny;
    }
    cp_async_wait_all();
    if (lane == 0) {
        // link x_{l0} -> x_{l0+1}
        ek += hl[wrap(cx - xs % L)] + hl[wrap(cy - xs / L)];
        atomicAdd(&st.meas[c].link_sum, double(ek) * chain_sign(st, c));
    }
}

}  // namespace hqmc

// local.cu -- local link updates of every worldline (Sec. 3.5.1, Eq. Rlocal), read in
// the position basis: slice l of a worldline moves one lattice step e (uniform over +x,
// -x, +y, -y) with its neighbours x_{l-1}, x_{l+1} held, accepted with probability
// min(1, R),
//     R = G(x' - x_{l-1}) W_l(x') G(x_{l+1} - x') / [G(x - x_{l-1}) W_l(x) G(x_{l+1} - x)],
// a handful of table lookups per move.  Slices of one colour (even l; odd l; l = M-1 alone
// when M is odd) are never neighbours in imaginary time, so one launch per colour updates
// all of them at once: one thread per (chain, worldline, slice of the colour), or with closed
// loops of one length both colours in one launch (local_pairs_kernel).  The kinetic link sums of
// the final paths are fused in; the occupancy histogram follows (local_hist_kernel).  With a
// permutation P at tau = beta, slice 0 of p follows slice M-1 of P^{-1}(p) and slice M-1
// of p precedes slice 0 of P(p) (other colours when M >= 2).
//
// The permutation update (Sec. 3.5.3) is here too: pair swaps of successors,
// P'(p) = P(q), P'(q) = P(p), accepted with probability min(1, R),
//     R = G(x_0^{P(q)} - x_{M-1}^p) G(x_0^{P(p)} - x_{M-1}^q)
//         / [G(x_0^{P(p)} - x_{M-1}^p) G(x_0^{P(q)} - x_{M-1}^q)],
// over disjoint pairs (2k + r, 2k + 1 + r) mod Nsig with a random rotation r, one thread
// per pair; every accepted swap flips the chain's sign.
#include <algorithm>

#include "device_common.cuh"
#include "internal.h"

namespace hqmc {

namespace {

constexpr int kLocalThreads = 256;
constexpr int kPairThreads = 320;  // most threads of local_pairs_kernel (160, 480 at M = 80: 244 us against 225)

__host__ __device__ inline int local_color(int M, int l) { return (M % 2 == 1 && l == M - 1) ? 2 : l % 2; }
// slices of colour c
__host__ __device__ inline int local_count(int M, int c) {
    if (M % 2 == 0) return c == 2 ? 0 : M / 2;
    return c == 2 ? 1 : (M - 1) / 2;
}

__device__ __forceinline__ int wrapd(int d, int L) { return d < 0 ? d + L : d; }

// G(b - a) = g(dx) g(dy), FP64
__device__ __forceinline__ double G2(const double *g, int L, int a, int b) {
    return g[wrapd(b % L - a % L, L)] * g[wrapd(b / L - a / L, L)];
}

// W_l(x) of worldline spin sg (Hirsch bit or Gaussian field), FP64
__device__ __forceinline__ double slice_w(const DevState &st, const ChainDev &cd, int sg, int l, int x) {
    const int L = cd.L;
    if (cd.gauss) return exp(cd.gcoup * st.gsig[cd.g_off + (long long)l * cd.N + x]);
    const int ix = x % L, iy = x / L;
    const uint32_t w = st.sbits[cd.s_off + ((long long)l * L + iy) * cd.wpl + (ix >> 5)];
    return ((w >> (ix & 31)) & 1u) ? cd.w_plus[sg] : cd.w_minus[sg];
}

// Per-chain tables of a CTA in shared memory, and division by L as a multiply-high (exact for
// sites below 2^14).
struct LocalTab {
    float g[kMaxL], h[kMaxL];
    float w[2][2];  // [spin][bit]
};
__device__ __forceinline__ void load_local_tab(LocalTab &t, const ChainDev &cd, const ChainTab &tb) {
    for (int j = threadIdx.x; j < cd.L; j += blockDim.x) {
        t.g[j] = tb.g_f[j];
        t.h[j] = tb.h_f[j];
    }
    if (threadIdx.x < 2) {
        t.w[threadIdx.x][0] = float(cd.w_minus[threadIdx.x]);
        t.w[threadIdx.x][1] = float(cd.w_plus[threadIdx.x]);
    }
    __syncthreads();
}
struct Site {
    int x, y;
};
__device__ __forceinline__ Site site_of(int s, int L, unsigned magic) {
    const int y = int(__umulhi(unsigned(s), magic));
    return {s - L * y, y};
}

// d/dt log G(b - a) from the FP32 link table (as the FFBS kernels)
__device__ __forceinline__ float link_h(const float *h, int L, Site a, Site b) {
    return h[wrapd(b.x - a.x, L)] + h[wrapd(b.y - a.y, L)];
}

// One move of slice l of a worldline at x between xm and xn, with the words of its step and its
// acceptance: returns the final site.  The decision u < R is the FP64 one.  FP32 decides it where u
// and R lie further apart than its error: the factors of the direction that does not move cancel
// (where they are so small that the FP64 products could underflow, FP64 decides), and four table
// values, their products and one division leave R within 2e-6 of itself, the leading 24 bits leave u
// within 2^-24.  All but about 1e-5 of the moves end there; the FP64 form took its
// 25 FP64 operations (two per cycle and SM) for every one.
__device__ __forceinline__ int local_move(const DevState &st, const ChainDev &cd, const ChainTab &tb, const LocalTab &lt, int sg,
                                          int l, int x, int xm, int xn, uint64_t wstep, uint64_t wacc, unsigned magic,
                                          bool &accepted) {
    const int L = cd.L, M = cd.M;
    const Site s = site_of(x, L, magic), a = site_of(xm, L, magic), b = site_of(xn, L, magic);
    const int dir = int(wstep >> 62);  // floor(4 u)
    Site n = s;
    if (dir == 0) n.x = s.x + 1 == L ? 0 : s.x + 1;
    else if (dir == 1) n.x = s.x == 0 ? L - 1 : s.x - 1;
    else if (dir == 2) n.y = s.y + 1 == L ? 0 : s.y + 1;
    else n.y = s.y == 0 ? L - 1 : s.y - 1;
    const int xnew = n.x + L * n.y;
    bool sure = false;
    if (!cd.gauss) {
        const uint32_t *rows = st.sbits + cd.s_off + (long long)l * L * cd.wpl;
        const uint32_t w0 = rows[s.y * cd.wpl + (s.x >> 5)], w1 = rows[n.y * cd.wpl + (n.x >> 5)];
        float num = lt.w[sg][(w1 >> (n.x & 31)) & 1u], den = lt.w[sg][(w0 >> (s.x & 31)) & 1u];
        float held = 1.f;  // the factors that cancel
        if (M > 1) {
            const bool ydir = dir >= 2;
            const int p = ydir ? s.y : s.x, q = ydir ? n.y : n.x, pa = ydir ? a.y : a.x, pb = ydir ? b.y : b.x;
            const int o = ydir ? s.x : s.y, oa = ydir ? a.x : a.y, ob = ydir ? b.x : b.y;
            held = lt.g[wrapd(o - oa, L)] * lt.g[wrapd(ob - o, L)];
            num *= lt.g[wrapd(q - pa, L)] * lt.g[wrapd(pb - q, L)];
            den *= lt.g[wrapd(p - pa, L)] * lt.g[wrapd(pb - p, L)];
        }
        const float R = num / den, u = float(uint32_t(wacc >> 40)) * 0x1.0p-24f;
        if (num > 1e-30f && den > 1e-30f && R < 1e30f && held > 1e-30f && held < 1e30f && fabsf(u - R) > 4e-6f * R + 1.2e-7f) {
            accepted = u < R;
            sure = true;
        }
    }
    if (!sure) {
        const double *g = tb.g_d;
        double R;
        if (M == 1) {
            // closed on itself (permutations need M >= 2): the link G(0) stays
            R = slice_w(st, cd, sg, l, xnew) / slice_w(st, cd, sg, l, x);
        } else {
            const double num = G2(g, L, xm, xnew) * slice_w(st, cd, sg, l, xnew) * G2(g, L, xnew, xn);
            const double den = G2(g, L, xm, x) * slice_w(st, cd, sg, l, x) * G2(g, L, x, xn);
            R = num / den;
        }
        accepted = u53(wacc) < R;
    }
    return accepted ? xnew : x;
}

// a warp's link sum and accepted moves
__device__ __forceinline__ void add_warp(const DevState &st, int c, float ek, int nacc) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ek += __shfl_xor_sync(0xffffffffu, ek, o);
    nacc = int(__reduce_add_sync(0xffffffffu, unsigned(nacc)));
    if ((threadIdx.x & 31) == 0) {
        if (ek != 0.f) atomicAdd(&st.meas[c].link_sum, double(ek) * chain_sign(st, c));
        if (nacc) atomicAdd(&st.meas[c].local_accepted, (unsigned long long)nacc);
    }
}

// One colour: one thread per (worldline, slice of the colour).
__global__ void __launch_bounds__(kLocalThreads) local_kernel(DevState st, int color) {
    const int c = blockIdx.y;
    const ChainDev &cd = st.chains[c];
    const int L = cd.L, M = cd.M, Nsig = cd.Nsig;
    const unsigned cnt = local_count(M, color), total = 2u * Nsig * cnt;
    if (blockIdx.x * blockDim.x >= total) return;
    __shared__ LocalTab lt;
    const ChainTab &tb = st.tabs[c];
    load_local_tab(lt, cd, tb);
    const unsigned u = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned magic = 0xffffffffu / unsigned(L) + 1u;
    float ek = 0.f;
    bool accepted = false;
    if (u < total) {
        const int wl = int(u / cnt), k = int(u - wl * cnt);
        const int l = color == 2 ? M - 1 : 2 * k + color;
        const int sg = wl / Nsig, p = wl - sg * Nsig;
        const int16_t *xspin = st.x + cd.x_off + (long long)sg * Nsig * M;
        int16_t *xp = st.x + cd.x_off + (long long)wl * M;
        const int lm = l == 0 ? M - 1 : l - 1, ln = l + 1 == M ? 0 : l + 1;
        const int *P = st.perm + cd.perm_off + sg * Nsig, *Pinv = P + 2 * Nsig;
        const int xm = l == 0 ? xspin[(long long)Pinv[p] * M + lm] : xp[lm];
        const int xn = l + 1 == M ? xspin[(long long)P[p] * M] : xp[ln];
        const int x = xp[l];
        // uniforms: phase 4, i = worldline, j = 2l (step) and 2l + 1 (acceptance)
        const u64x4 w4 = philox4x64_10((uint64_t)(l >> 1), (uint64_t)wl, 4, *st.sweep, cd.seed, 0);
        const int xf = local_move(st, cd, tb, lt, sg, l, x, xm, xn, (l & 1) ? w4.v[2] : w4.v[0],
                                  (l & 1) ? w4.v[3] : w4.v[1], magic, accepted);
        if (accepted) xp[l] = int16_t(xf);
        // kinetic links whose other end is already final (a lower colour); M = 1: the self link
        const Site a = site_of(xm, L, magic), f = site_of(xf, L, magic), b = site_of(xn, L, magic);
        if (M == 1) {
            ek = link_h(lt.h, L, f, f);
        } else {
            if (local_color(M, lm) < color) ek += link_h(lt.h, L, a, f);
            if (local_color(M, ln) < color) ek += link_h(lt.h, L, f, b);
        }
    }
    add_warp(st, c, ek, accepted ? 1 : 0);
}

// Colours 0 and 1 of closed loops in one launch (no permutation in use, so a worldline's neighbours
// in imaginary time are its own slices): a CTA holds W whole worldlines in shared memory, and the
// thread of the pair (l, l + 1), l even, moves l, waits for the others, and moves l + 1 with the
// other half of the same Philox block.  A colour each (three launches, the last one empty at even M)
// drew every block twice and read the neighbours from memory.  W makes the CTA's pairs whole warps,
// so that the FP32 link sums group the slices as a launch per colour does.
__global__ void __launch_bounds__(kPairThreads) local_pairs_kernel(DevState st, int W) {
    extern __shared__ int16_t xs[];  // [W][M]
    __shared__ LocalTab lt;
    const int c = blockIdx.y;
    const ChainDev &cd = st.chains[c];
    const int L = cd.L, M = cd.M, Nsig = cd.Nsig;
    const int cnt = local_count(M, 0);
    const int wl0 = blockIdx.x * W, nw = min(W, 2 * Nsig - wl0);
    if (nw <= 0 || cnt == 0) return;
    const ChainTab &tb = st.tabs[c];
    load_local_tab(lt, cd, tb);
    const unsigned magic = 0xffffffffu / unsigned(L) + 1u;
    int16_t *xg = st.x + cd.x_off + (long long)wl0 * M;
    for (int k = threadIdx.x; k < nw * M; k += blockDim.x) xs[k] = xg[k];
    __syncthreads();
    const uint64_t sweep = *st.sweep;
    const int items = nw * cnt, rounds = (W * cnt + int(blockDim.x) - 1) / int(blockDim.x);
    uint64_t wd2 = 0, wd3 = 0;
    for (int color = 0; color < 2; ++color) {
        for (int r = 0; r < rounds; ++r) {
            const int it = r * blockDim.x + threadIdx.x;
            float ek = 0.f;
            bool accepted = false;
            if (it < items) {
                const int w = it / cnt, k = it - w * cnt, l = 2 * k + color;
                const int wl = wl0 + w, sg = wl / Nsig;
                int16_t *xp = xs + w * M;
                const int lm = l == 0 ? M - 1 : l - 1, ln = l + 1 == M ? 0 : l + 1;
                const int xm = xp[lm], xn = xp[ln];
                uint64_t ws = wd2, wa = wd3;
                if (color == 0 || rounds > 1) {
                    const u64x4 w4 = philox4x64_10((uint64_t)k, (uint64_t)wl, 4, sweep, cd.seed, 0);
                    wd2 = w4.v[2];
                    wd3 = w4.v[3];
                    ws = color ? wd2 : w4.v[0];
                    wa = color ? wd3 : w4.v[1];
                }
                const int xf = local_move(st, cd, tb, lt, sg, l, xp[l], xm, xn, ws, wa, magic, accepted);
                if (accepted) xp[l] = int16_t(xf);
                if (color) {
                    const Site a = site_of(xm, L, magic), f = site_of(xf, L, magic), b = site_of(xn, L, magic);
                    ek += link_h(lt.h, L, a, f);
                    if (local_color(M, ln) == 0) ek += link_h(lt.h, L, f, b);
                }
            }
            if (r * int(blockDim.x) + int(threadIdx.x & ~31u) < items) add_warp(st, c, ek, accepted ? 1 : 0);
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < nw * M; k += blockDim.x) xg[k] = xs[k];
}

__global__ void __launch_bounds__(kLocalThreads) perm_kernel(DevState st) {
    const int c = blockIdx.y, sg = blockIdx.z;
    const ChainDev &cd = st.chains[c];
    const int L = cd.L, M = cd.M, Nsig = cd.Nsig, npr = Nsig / 2;
    const uint64_t sweep = *st.sweep;
    // pairing rotation (phase 5, i = sigma, j = 0)
    int r = int(u53(philox4x64_10(0, (uint64_t)sg, 5, sweep, cd.seed, 0).v[0]) * Nsig);
    if (r >= Nsig) r = Nsig - 1;
    int *P = st.perm + cd.perm_off + sg * Nsig, *Pinv = P + 2 * Nsig;
    const int16_t *X = st.x + cd.x_off + (long long)sg * Nsig * M;
    const double *g = st.tabs[c].g_d;
    unsigned cnt = 0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < npr; k += gridDim.x * blockDim.x) {
        int p = 2 * k + r, q = 2 * k + 1 + r;
        if (p >= Nsig) p -= Nsig;
        if (q >= Nsig) q -= Nsig;
        const int Pp = P[p], Pq = P[q];
        const int xlp = X[(long long)p * M + M - 1], xlq = X[(long long)q * M + M - 1];
        const int a0 = X[(long long)Pp * M], b0 = X[(long long)Pq * M];
        const double R = (G2(g, L, xlp, b0) * G2(g, L, xlq, a0)) / (G2(g, L, xlp, a0) * G2(g, L, xlq, b0));
        // pair k: phase 5, i = sigma, j = 1 + k
        const u64x4 w4 = philox4x64_10((uint64_t)((1 + k) >> 2), (uint64_t)sg, 5, sweep, cd.seed, 0);
        const int wsel = (1 + k) & 3;
        const double u = u53(wsel == 0 ? w4.v[0] : wsel == 1 ? w4.v[1] : wsel == 2 ? w4.v[2] : w4.v[3]);
        if (u < R) {
            P[p] = Pq;
            P[q] = Pp;
            Pinv[Pq] = p;
            Pinv[Pp] = q;
            ++cnt;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if ((threadIdx.x & 31) == 0 && cnt) {
        atomicAdd(&st.meas[c].perm_accepted, (unsigned long long)cnt);
        if (cnt & 1u) atomicXor(&st.parity[c], 1u);
    }
}

// Occupancy histogram of the new worldlines: a CTA counts S slices of one spin in shared memory and
// writes them out.  An atomic per move into global memory took 105 of 244 us (64 chains of L = 32:
// 5.2 million scattered reductions), this 26.
__global__ void __launch_bounds__(kLocalThreads) local_hist_kernel(DevState st, int S) {
    extern __shared__ int cnt[];  // [S][N]
    const ChainDev &cd = st.chains[blockIdx.y];
    const int N = cd.N, M = cd.M, Nsig = cd.Nsig, sg = blockIdx.z;
    const int l0 = blockIdx.x * S;
    if (l0 >= M) return;
    const int ns = min(S, M - l0);
    for (int k = threadIdx.x; k < ns * N; k += blockDim.x) cnt[k] = 0;
    __syncthreads();
    const int16_t *x = st.x + cd.x_off + (long long)sg * Nsig * M + l0;
    // consecutive threads take the slices of one worldline, then the next worldline's
    for (int k = threadIdx.x; k < Nsig * ns; k += blockDim.x) {
        const int p = k / ns, s = k - p * ns;
        atomicAdd(&cnt[s * N + x[(long long)p * M + s]], 1);
    }
    __syncthreads();
    int *h = st.hist + cd.h_off + ((long long)sg * M + l0) * N;
    for (int k = threadIdx.x; k < ns * N; k += blockDim.x) h[k] = cnt[k];
}

}  // namespace

cudaError_t launch_perm(const DevState &st, int nchains, int max_pairs, cudaStream_t stream) {
    if (max_pairs <= 0) return cudaSuccess;
    const dim3 grid(std::min((max_pairs + kLocalThreads - 1) / kLocalThreads, 64), nchains, 2);
    perm_kernel<<<grid, kLocalThreads, 0, stream>>>(st);
    return cudaGetLastError();
}

// worldlines per CTA of local_pairs_kernel: whole warps of pairs, a thread each up to kPairThreads;
// 0 where they would not fit its shared memory
static int local_pairs_wl(int M) {
    const int cnt = local_count(M, 0);
    if (cnt == 0) return 1;
    int unit = 32;  // 32 / gcd(cnt, 32)
    for (int c = cnt; unit > 1 && c % 2 == 0; c /= 2) unit /= 2;
    const int W = unit * std::max(1, kPairThreads / (unit * cnt));
    return size_t(W) * M * 2 <= 40 * 1024 ? W : 0;
}

cudaError_t launch_local(const DevState &st, const LocalShape *chains, int nchains, bool closed, cudaStream_t stream) {
    // one value of W for the launch: chains of one M (the usual batch) take the fused form
    bool same = closed && nchains > 0;
    int most_wl = 0;
    for (int i = 0; i < nchains; ++i) {
        same = same && chains[i].M == chains[0].M;
        most_wl = std::max(most_wl, 2 * chains[i].Nsig);
    }
    const int W = same ? local_pairs_wl(chains[0].M) : 0;
    int first = 0;
    if (W > 0) {
        if (local_count(chains[0].M, 0) > 0)
            local_pairs_kernel<<<dim3((most_wl + W - 1) / W, nchains), std::min(kPairThreads, W * local_count(chains[0].M, 0)),
                                 size_t(W) * chains[0].M * 2, stream>>>(st, W);
        first = 2;
    }
    for (int color = first; color < 3; ++color) {
        long long units = 0;
        for (int i = 0; i < nchains; ++i)
            units = std::max(units, 2LL * chains[i].Nsig * local_count(chains[i].M, color));
        if (units == 0) continue;
        local_kernel<<<dim3(int((units + kLocalThreads - 1) / kLocalThreads), nchains), kLocalThreads, 0, stream>>>(st, color);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int max_M = 0, max_N = 0;
    for (int i = 0; i < nchains; ++i) {
        max_M = std::max(max_M, chains[i].M);
        max_N = std::max(max_N, chains[i].N);
    }
    // 8 slices (32 KB) up to L = 32; one slice of L = 128 takes 64 KB
    const int S = std::max(1, std::min(8, 8192 / max_N));
    const size_t sm = size_t(S) * max_N * 4;
    if (sm > 48 * 1024) {
        e = cudaFuncSetAttribute(local_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm));
        if (e != cudaSuccess) return e;
    }
    local_hist_kernel<<<dim3((max_M + S - 1) / S, nchains, 2), kLocalThreads, sm, stream>>>(st, S);
    return cudaGetLastError();
}

}  // namespace hqmc

// Level-2 approximation (§4.5): after the level-1 delegate cut and thin skin,
// every b x b block of sites is cut exactly on its own, the pairs that leave
// the block taken against the neighbours' current labels, blocks updated in a
// two-colour order (see gs_block_descent in gazecut.h).
//
// A block problem is tiny (b <= 3: at most 3 x 3 sites, at most 3b labels in
// the skin), so one warp solves it exactly by min-sum dynamic programming over
// the block's rows: a row state is the labels of the row's sites (n^bw states
// for n labels), the row cost holds the sites' data and border terms and the
// pairs inside the row, and the pairs between consecutive rows -- a sum over
// the columns -- are applied one column at a time (a min-plus transform of one
// label digit).  The transform is linear in n: h~ is the min-plus convolution
// of lambda |d| on |d| <= 1 (infinite beyond) with (lambda + inhibit) |d|, so a
// line of n labels takes a three-point minimum and one running minimum each
// way.  Moving from row to row costs 2 bw n^bw steps, instead of n^(2 bw) for
// all pairs of states or bw n^(bw+1) for all pairs of labels.  Forward and
// backward passes give every row state's min-marginal; the smallest label a site
// takes in any minimiser, read from the states whose min-marginal equals the
// minimum, is the site's label in the component-wise smallest minimiser (the
// minimisers of this convex-prior energy form a lattice under component-wise
// min), the same canonical answer as the minimal source set of the block's cut.
#include "gs_internal.cuh"

namespace gs {

constexpr int kL2Warps = 4;                       // warps (blocks in flight) per CTA
constexpr long long kL2Inf = 1ll << 50;           // data term outside a site's bounds

__device__ __forceinline__ long long htil(int d, long long lam, long long inh) {
    const long long a = d < 0 ? -d : d;
    return lam * a + (a > 1 ? inh * (a - 1) : 0);
}

struct L2Args {
    const int32_t *cost;    // [h][n_g][D]
    const int32_t *lo, *hi; // [h][n_g]
    int32_t *labels;        // [h][n_g], updated in place for the blocks of one colour
    int32_t *status;
    int ng, h, D, b, colour, nbx, nby, scap;
    long long lam, h2h, h2v;
};

// Min-plus transform of one label digit of every row state (states whose other
// digits agree lie pw apart, n of them: a line): out = min over d of in(d) +
// h~_v(d - digit), in place when in == out.  One line a lane: the lane holds
// the line's previous inputs, so it may overwrite them.
__device__ __forceinline__ void col_transform(const long long *in, long long *out, int lines, int n,
                                              unsigned rn, int pw, bool top, long long lam,
                                              long long inh, int lane) {
    for (int q = lane; q < lines; q += 32) {
        // the line's first state: q with a digit 0 put in at pw
        const int hi = pw == 1 ? q : top ? 0 : n == 1 ? q : (int)__umulhi((unsigned)q, rn);
        const int base = pw == 1 ? q * n : q - hi * pw + hi * pw * n;
        long long cur = in[base], prev = kL2Inf * 64, run = kL2Inf * 64;
        for (int d = 0; d < n; d++) {
            const long long next = d + 1 < n ? in[base + (d + 1) * pw] : kL2Inf * 64;
            const long long m = min(cur, min(prev, next) + lam);
            run = min(m, run + lam + inh);
            out[base + d * pw] = run;
            prev = cur;
            cur = next;
        }
        for (int d = n - 2; d >= 0; d--) {
            run = min(out[base + d * pw], run + lam + inh);
            out[base + d * pw] = run;
        }
    }
    __syncwarp();
}

// One warp per block.  Bound by the latency of the lines' running minima and
// by how many warps hide it: 4 S + 96 words of 8 bytes a warp (S row states, 729
// for 3 x 3 sites and 9 labels) leave room for eight warps per SM.  384x288x16
// at b = 3, four half-passes over 11,000 blocks: 4.37 ms with the transform over
// all pairs of labels and its own two buffers (four warps per SM), 0.90 ms now.
__global__ void __launch_bounds__(32 * kL2Warps) k_block_descent(const L2Args a) {
    extern __shared__ long long l2sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S_cap = a.scap;
    long long *F = l2sm + (size_t)warp * (4 * S_cap + 96);   // F[3][S_cap]
    long long *Bk = F + 3 * S_cap;
    long long *U = Bk + S_cap;                                 // [bh][bw][n], at most 96
    // the colour's blocks: n_even in an even row of blocks, nbx in two rows
    const int n_even = (a.nbx + 1 - a.colour) / 2;
    const int nblocks = a.nby / 2 * a.nbx + (a.nby & 1) * n_even;
    for (int k = blockIdx.x * kL2Warps + warp; k < nblocks; k += gridDim.x * kL2Warps) {
        const int pair = k / a.nbx, rest = k - pair * a.nbx, odd = rest >= n_even;
        const int by = 2 * pair + odd, bx = 2 * (rest - odd * n_even) + ((by + a.colour) & 1);
        const int y0 = by * a.b, W0 = bx * a.b;
        const int bh = min(a.b, a.h - y0), bw = min(a.b, a.ng - W0);
        // the block's label range: the union of its sites' bounds
        int LO = a.D, HI = -1, bad = 0;
        for (int t = lane; t < bh * bw; t += 32) {
            const int64_t v = (int64_t)(y0 + t / bw) * a.ng + W0 + t % bw;
            const int l = a.lo[v], u = a.hi[v];
            bad |= l < 0 || l > u || u > a.D - 1;
            LO = min(LO, l);
            HI = max(HI, u);
        }
        for (int o = 16; o > 0; o >>= 1) {
            LO = min(LO, __shfl_xor_sync(0xffffffffu, LO, o));
            HI = max(HI, __shfl_xor_sync(0xffffffffu, HI, o));
            bad |= __shfl_xor_sync(0xffffffffu, bad, o);
        }
        const int n = HI - LO + 1;
        int S = 1;
        for (int c = 0; c < bw && !bad; c++) {
            if (S > S_cap / max(n, 1)) bad = 1;
            S *= n;
        }
        if (bad || n < 1 || bh * bw * n > 96) {
            if (lane == 0) atomicCAS(a.status, GS_OK, GS_ERR_INVAL);
            continue;
        }
        const unsigned rn = n > 1 ? (unsigned)((0x100000000ull + n - 1) / n) : 0u;   // for s / n
        // unary terms: data term inside the site's bounds, plus the pairs to
        // sites outside the block against their current labels
        for (int t = lane; t < bh * bw * n; t += 32) {
            const int kk = t % n, c = (t / n) % bw, r = t / (n * bw);
            const int y = y0 + r, W = W0 + c, l = LO + kk;
            const int64_t v = (int64_t)y * a.ng + W;
            long long u;
            if (l < a.lo[v] || l > a.hi[v]) {
                u = kL2Inf;
            } else {
                u = a.cost[v * a.D + l];
                if (W == W0 && W > 0) u += htil(l - a.labels[v - 1], a.lam, a.h2h);
                if (W == W0 + bw - 1 && W < a.ng - 1) u += htil(l - a.labels[v + 1], a.lam, a.h2h);
                if (y == y0 && y > 0) u += htil(l - a.labels[v - a.ng], a.lam, a.h2v);
                if (y == y0 + bh - 1 && y < a.h - 1) u += htil(l - a.labels[v + a.ng], a.lam, a.h2v);
            }
            U[t] = u;
        }
        __syncwarp();
        // row cost of state s in row r (data, border terms, pairs inside the row)
        auto row_cost = [&](int r, int s) {
            long long acc = 0;
            int prev = 0;
            for (int c = 0; c < bw; c++) {
                const int q = n > 1 ? (int)__umulhi((unsigned)s, rn) : s;
                const int d = s - q * n;
                s = q;
                acc += U[(r * bw + c) * n + d];
                if (c > 0) acc += htil(prev - d, a.lam, a.h2h);
                prev = d;
            }
            return acc;
        };
        // min-plus step to the next row, digit by digit, from src into dst
        auto row_step = [&](const long long *src, long long *dst) {
            int pw = 1;
            for (int c = 0; c < bw; c++, pw *= n)
                col_transform(c == 0 ? src : dst, dst, S / n, n, rn, pw, c == bw - 1, a.lam, a.h2v,
                              lane);
        };
        // forward
        for (int s = lane; s < S; s += 32) F[s] = row_cost(0, s);
        __syncwarp();
        for (int r = 1; r < bh; r++) {
            long long *Fr = F + r * S_cap;
            row_step(F + (r - 1) * S_cap, Fr);
            for (int s = lane; s < S; s += 32) Fr[s] += row_cost(r, s);
            __syncwarp();
        }
        // minimum energy of the block problem
        long long Emin = kL2Inf * 64;
        for (int s = lane; s < S; s += 32) Emin = min(Emin, F[(bh - 1) * S_cap + s]);
        for (int o = 16; o > 0; o >>= 1) Emin = min(Emin, __shfl_xor_sync(0xffffffffu, Emin, o));
        // backward, with the smallest label of every site among the minimisers
        for (int s = lane; s < S; s += 32) Bk[s] = 0;
        __syncwarp();
        for (int r = bh - 1; r >= 0; r--) {
            if (r < bh - 1) {
                // Bk_r(s) = min over s' of V(s, s') + R_(r+1)(s') + Bk_(r+1)(s')
                for (int s = lane; s < S; s += 32) Bk[s] += row_cost(r + 1, s);
                __syncwarp();
                row_step(Bk, Bk);
            }
            int best[3] = {n, n, n};             // bw <= 3
            for (int s = lane; s < S; s += 32) {
                if (F[r * S_cap + s] + Bk[s] != Emin) continue;
                int rest = s;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const int q = n > 1 ? (int)__umulhi((unsigned)rest, rn) : rest;
                    best[c] = min(best[c], rest - q * n);
                    rest = q;
                }
            }
#pragma unroll
            for (int c = 0; c < 3; c++) best[c] = __reduce_min_sync(0xffffffffu, best[c]);
            if (lane < bw) {
                const int d = lane == 0 ? best[0] : lane == 1 ? best[1] : best[2];
                const int64_t v = (int64_t)(y0 + r) * a.ng + W0 + lane;
                if (d < n) a.labels[v] = LO + d;
                else atomicCAS(a.status, GS_OK, GS_ERR_LABELS);
            }
            __syncwarp();
        }
    }
}

// Start labels: each site's first argmin of the data term inside its
// delegate's depth bin [b Xc, min(b Xc + b, D) - 1].
__global__ void k_level2_start(const int32_t *__restrict__ cost, const int32_t *__restrict__ Xc,
                               int ng, int h, int D, int b, int ngc, int Dc,
                               int32_t *__restrict__ labels, int32_t *status) {
    int bad = 0;
    const int64_t sites = (int64_t)ng * h;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < sites;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int W = (int)(v % ng), y = (int)(v / ng);
        const int Lc = Xc[(int64_t)(y / b) * ngc + W / b];
        if (Lc < 0 || Lc >= Dc) {
            bad = 1;
            labels[v] = 0;
            continue;
        }
        const int a0 = b * Lc, z = min(a0 + b, D);
        int best = a0;
        int32_t bc = cost[v * D + a0];
        for (int l = a0 + 1; l < z; l++) {
            const int32_t c = cost[v * D + l];
            if (c < bc) {
                bc = c;
                best = l;
            }
        }
        labels[v] = best;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicCAS(status, GS_OK, GS_ERR_LABELS);
}

// Row states a block of b x b sites may need: (labels of the skin)^b.
static int state_cap(int b, int D) {
    const int n = std::min(3 * b, D);
    int S = 1;
    for (int c = 0; c < b; c++) S *= n;
    return S;
}

}  // namespace gs

using namespace gs;

extern "C" int gs_level2_start(const int32_t *cost, const gs_params *p, int32_t b,
                               const int32_t *coarse_labels, int32_t *labels, int32_t *status,
                               void *stream) {
    Geom g;
    if (make_geom(p, &g) != GS_OK || !cost || !coarse_labels || !labels || !status)
        return GS_ERR_INVAL;
    if (b < 1 || b >= g.D) return GS_ERR_INVAL;
    const int ngc = (g.ng + b - 1) / b, Dc = (g.D + b - 1) / b;
    const int64_t sites = (int64_t)g.ng * g.h;
    k_level2_start<<<grid_for(sites, 16), 256, 0, (cudaStream_t)stream>>>(
        cost, coarse_labels, g.ng, g.h, g.D, b, ngc, Dc, labels, status);
    count_launches(1);
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

extern "C" int gs_block_descent(const int32_t *cost, const gs_params *p, int32_t b,
                                const int32_t *lo, const int32_t *hi, int32_t *labels,
                                int32_t passes, int32_t *status, void *stream) {
    Geom g;
    if (make_geom(p, &g) != GS_OK || !cost || !lo || !hi || !labels || !status)
        return GS_ERR_INVAL;
    if (b < 1 || b > 3 || passes < 0) return GS_ERR_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    L2Args a;
    a.cost = cost;
    a.lo = lo;
    a.hi = hi;
    a.labels = labels;
    a.status = status;
    a.ng = g.ng;
    a.h = g.h;
    a.D = g.D;
    a.b = b;
    a.nbx = (g.ng + b - 1) / b;
    a.nby = (g.h + b - 1) / b;
    a.scap = state_cap(b, g.D);
    a.lam = g.lam;
    a.h2h = g.h2h;
    a.h2v = g.h2v;
    const size_t smem = (size_t)kL2Warps * (4 * a.scap + 96) * sizeof(long long);
    GS_CUDA_TRY(cudaFuncSetAttribute(k_block_descent, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    const int64_t half = ((int64_t)a.nbx * a.nby + 1) / 2;
    const int grid = (int)std::max<int64_t>(
        1, std::min<int64_t>((half + kL2Warps - 1) / kL2Warps, 4 * (int64_t)device_sms()));
    for (int it = 0; it < passes; it++) {
        for (int colour = 0; colour < 2; colour++) {
            a.colour = colour;
            k_block_descent<<<grid, 32 * kL2Warps, smem, st>>>(a);
            count_launches(1);
        }
    }
    GS_CUDA_TRY(cudaGetLastError());
    return GS_OK;
}

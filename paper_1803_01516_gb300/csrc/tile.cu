// Persistent, tiled push-relabel with global relabelling (§4.4) for the chain
// graph of §3 / Fig. 4.
//
// One cooperative launch runs the whole solve.  The node grid is cut into
// tiles of TW sites x TH rows x all K chain layers (whole chains, so the data
// arcs and their infinite reverse arcs never leave a tile).  A CTA stages a
// tile plus a one-site halo in shared memory and works on it locally; tiles
// exchange flow only through atomics on global memory, and a pair's steps
// (see "the solve loop" below) separate its phases:
//
//   global relabel  heights = breadth-first distance to the nearest node with
//                   sink capacity left, computed as a monotone relaxation:
//                   every tile relaxes to its local fixed point in shared
//                   memory, passes repeat until a whole pass changes nothing
//                   (the exact distances); the pass also counts active nodes
//                   (positive excess, finite height); zero active nodes means
//                   the preflow is maximum and the solve ends.
//   sweep rounds    every tile with active nodes runs up to `local_iters`
//                   push/relabel iterations in shared memory, and writes its
//                   changes -- its own words and what it pushed into its halo
//                   -- back as deltas, so concurrent tiles compose.
//
// Correctness does not depend on the interleaving: every push moves at most
// the excess and the residual its tile can see, and both only grow under
// other tiles' updates, so the state stays a valid preflow; heights only steer
// pushes.  The exit test is the exact reachability computed by the relabel.
#include <cstring>
#include <mutex>

#include "arcs.cuh"

namespace gs {

constexpr int kTileThreads = 512;            // threads per block (256 on request: two per SM)
constexpr int kInitOuter = 8;                 // relaxation rounds of a first relabel pass
constexpr int kBlk = 4;                       // chain layers of a thread's block of own nodes

struct TileGeom {
    int TW, TH;        // sites per tile along W and y
    int SJ;            // shared-memory stride of one field of one chain layer: TW + 2
    int SYs;           // shared-memory stride of one row of sites: (K + 1) * 9 * SJ, padded
                       // so that a warp's lanes fall on different banks
    int words;         // shared words of a tile: (TH + 2) rows and kBlk layers
    int S, nblk;       // sites of a tile, blocks of kBlk layers of a chain
    int TN;            // own nodes per tile S * K
    unsigned rTH, rS;  // ceil(2^32 / TH) (0 when TH = 1) and ceil(2^32 / S), for divisions
    int tiles_w, tiles_h, T;
};

struct SolveArgs {
    Geom g;
    TileGeom t;
    State s;
    uint16_t *amask;     // per node: residual-arc bits (14) | has-excess bit (15)
    int32_t *tile_act;   // [2][T] tiles with work in the current / next sweep round
    int32_t *tile_dirty; // [2][T] tiles whose halo heights changed in the last relabel pass
    int32_t *tile_cnt;   // [T] active nodes per tile after its last relabel pass
    int32_t *tile_list;  // [3][T] tiles queued for a step (slot = step mod 3)
    int32_t *hgt;        // distances the relabel passes compute (state heights, or marks)
    int dir;             // 0: distance to sink capacity over out-arcs (heights);
                         // 1: distance from positive excess over in-arcs (reachability);
                         // 2: label extraction of an exact solve, 1 unless the state is
                         //    the label-reversed problem, then 0
    Ctrl *ctrl;          // the pair's control block (statistics)
    int32_t *status;     // the caller's device status word
    int32_t *labels;     // label extraction output [h][n_g]
    int64_t *flow;       // label extraction output [1]
    int mode, sweeps_per_relabel, local_iters, relabel_passes, tail_iters;
    long long fixed_sweeps, max_iters;
    int tpt;             // blocks of own nodes per thread of the pair's tile shape (1 or 2)
};

// Every read of solver state inside the persistent kernel bypasses L1: other
// SMs update the same words during the launch, and L1 is not coherent.
template <class T>
__device__ __forceinline__ T ld(const T *p) { return __ldcg(p); }

// Block-wide sum (all threads get the total).
__device__ __forceinline__ long long block_sum(long long v) {
    __shared__ unsigned long long s_sum;
    __syncthreads();
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    if (v) atomicAdd(&s_sum, (unsigned long long)v);
    __syncthreads();
    return (long long)s_sum;
}

__device__ __forceinline__ bool aborted(Ctrl *ctrl) {
    return *(volatile int32_t *)&ctrl->abort != 0;
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Atomics with acquire / release semantics at GPU scope (one instruction in
// place of a fence and a relaxed atomic).
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned *p, unsigned v) {
    unsigned r;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(r) : "l"(p), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ unsigned long long atom_add_acquire(unsigned long long *p,
                                                             unsigned long long v) {
    unsigned long long r;
    asm volatile("atom.acquire.gpu.global.add.u64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(v) : "memory");
    return r;
}
__device__ __forceinline__ unsigned long long atom_add_relaxed(unsigned long long *p,
                                                             unsigned long long v) {
    unsigned long long r;
    asm volatile("atom.relaxed.gpu.global.add.u64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(v) : "memory");
    return r;
}
__device__ __forceinline__ void red_add_release(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long atom_exch_release(unsigned long long *p,
                                                              unsigned long long v) {
    unsigned long long r;
    asm volatile("atom.release.gpu.global.exch.b64 %0, [%1], %2;" : "=l"(r) : "l"(p), "l"(v) : "memory");
    return r;
}

// ------------------------------------------------------- tile addressing ---
//
// A tile in shared memory: rows of sites (TH own rows and one halo row on
// either side), in a row its K chain layers, in a layer the nine fields, in a
// field TW + 2 sites.  The offsets from a node's cell to its 14 neighbours and
// to the words of its arcs are then compile-time constants (tile width TWC)
// around three addresses -- the node's cell, the one a row up and the one a
// row down -- and go into the load instructions.  With one array per field
// they were 28 run-time offsets, each an add and, for arcs that may not
// exist, a select.  Between the rows lies a layer of padding whose words all
// hold kInfH (build_tables): the layers past a chain's ends have infinite
// heights, like the positions outside the grid, so an arc that does not exist
// is never admissible and never gives a minimum, whatever its residual reads.
// A thread's own nodes are blocks of kBlk consecutive layers of one site:
// block n of a tile (n = threadIdx.x, and threadIdx.x + blockDim.x when a tile
// has more blocks than threads) is site n mod S, layers kBlk (n / S) onwards,
// so a warp's lanes are neighbouring sites of one row of blocks.

enum { F_EX = 0, F_HT, F_RC, F_RR, F_RD, F_I0, F_I1, F_I2, F_I3, F_N };

// Strides of a tile whose width is TWC at compile time (0: at run time).
template <int TWC>
struct Lay {
    int sy, sj_;
    __device__ __forceinline__ explicit Lay(const TileGeom &t) : sy(t.SYs), sj_(t.SJ) {}
    __device__ __forceinline__ int sj() const { return TWC ? TWC + 2 : sj_; }
    // word offset of field f at (dj, dw) from a cell of the same row
    __device__ __forceinline__ int at(int f, int dj = 0, int dw = 0) const {
        return (f + F_N * dj) * sj() + dw;
    }
    // cell of tile position (yl, j, wl), yl in [-1, TH], wl in [-1, TW]
    __device__ __forceinline__ int cell(int yl, int j, int wl) const {
        return (yl + 1) * sy + (j + 1) * F_N * sj() + (wl + 1);
    }
};

template <int TWC>
__device__ __forceinline__ int tile_w(const TileGeom &t) { return TWC ? TWC : t.TW; }

// Residuals of the 14 slots of cell c (anything for an arc that does not
// exist: its head's height is infinite).
template <int TWC>
__device__ __forceinline__ void load_residuals(const Lay<TWC> &l, const Geom &g,
                                               const volatile int32_t *c,
                                               int32_t (&r)[kSlots]) {
    const volatile int32_t *u = c - l.sy, *d = c + l.sy;
    r[0] = c[l.at(F_RC)];
    r[1] = kInfR;
    r[2] = c[l.at(F_RR)];
    r[3] = g.lam2 - c[l.at(F_RR, 0, -1)];
    r[4] = c[l.at(F_RD)];
    r[5] = g.lam2 - u[l.at(F_RD)];
    r[6] = c[l.at(F_I0)];
    r[7] = c[l.at(F_I1)];
    r[8] = c[l.at(F_I2)];
    r[9] = c[l.at(F_I3)];
    r[10] = g.h2h - c[l.at(F_I1, 1, -1)];
    r[11] = g.h2h - c[l.at(F_I0, 1, 1)];
    r[12] = g.h2v - u[l.at(F_I3, 1)];
    r[13] = g.h2v - d[l.at(F_I2, 1)];
}

// Fire-and-forget adds (PTX red): no result comes back, so a push does not
// wait for the memory system before the next one.
__device__ __forceinline__ void red_add_smem(int32_t *p, int32_t v) {
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)),
                 "r"(v));
}
// Shared memory by 32-bit address, under a predicate: a discharge has no
// branches (each took longer than the access it guarded).
__device__ __forceinline__ int32_t lds(unsigned a) {
    int32_t r;
    asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(r) : "r"(a));
    return r;
}
__device__ __forceinline__ void sts(unsigned a, int32_t v) {
    asm volatile("st.volatile.shared.s32 [%0], %1;" ::"r"(a), "r"(v));
}
__device__ __forceinline__ void sts16(unsigned a, int v) {
    asm volatile("{ .reg .b16 h; cvt.u16.u32 h, %1; st.volatile.shared.u16 [%0], h; }" ::"r"(a),
                 "r"(v));
}
__device__ __forceinline__ int32_t atom_add_nz(unsigned a, int32_t v) {
    int32_t r;
    asm volatile("{ .reg .pred q; setp.ne.s32 q, %2, 0; mov.s32 %0, 0;"
                 "  @q atom.shared.add.s32 %0, [%1], %2; }" : "=&r"(r) : "r"(a), "r"(v));
    return r;
}
// Store w at a where p is not 0, and add v to the word at b if it is not 0;
// returns what b held before (0 if it was left alone).
__device__ __forceinline__ int32_t push_words(unsigned a, int32_t w, int32_t p, unsigned b,
                                              int32_t v) {
    int32_t r;
    asm volatile("{ .reg .pred p, q; setp.ne.s32 p, %3, 0; setp.ne.s32 q, %5, 0; mov.s32 %0, 0;"
                 "  @p st.volatile.shared.s32 [%1], %2; @q atom.shared.add.s32 %0, [%4], %5; }"
                 : "=&r"(r) : "r"(a), "r"(w), "r"(p), "r"(b), "r"(v));
    return r;
}
// Add v to a global word unless it is 0, and store v where p holds: no branch.
__device__ __forceinline__ void red_add_nz(int32_t *a, int32_t v) {
    asm volatile("{ .reg .pred p; setp.ne.s32 p, %1, 0;"
                 "  @p red.relaxed.gpu.global.add.s32 [%0], %1; }" ::"l"(a), "r"(v));
}
__device__ __forceinline__ void stg_if(bool p, int32_t *a, int32_t v) {
    asm volatile("{ .reg .pred p; setp.ne.s32 p, %2, 0; @p st.global.cg.s32 [%0], %1; }" ::"l"(a),
                 "r"(v), "r"((int)p));
}
__device__ __forceinline__ void red_add_gmem(int32_t *p, int32_t v) {
    asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v));
}

struct TileOrigin {
    int tx, ty, W0, y0;
};

__device__ __forceinline__ TileOrigin tile_origin(const TileGeom &t, int tile) {
    TileOrigin o;
    o.tx = tile % t.tiles_w;
    o.ty = tile / t.tiles_w;
    o.W0 = o.tx * t.TW;
    o.y0 = o.ty * t.TH;
    return o;
}

// Staging with every global load issued before any shared-memory store: a
// thread's first two halo cells go through registers (HaloRegs), so the halo
// and the own nodes of a tile arrive in one round trip to L2 instead of one
// per loop.  Cells past the first 2 x blockDim (large depth ranges) are
// loaded afterwards by halo_rest.
struct HaloRegs {
    int32_t h[2], r1[2], r2[2];
    int cell[2], kind[2];      // kind -1: no cell
};

// Halo cell n of the combined index space: the left and right columns
// (2 TH K cells), then the top and bottom rows (2 K TW cells).  kind 0..3 =
// left, right, top, bottom.
template <int TWC>
__device__ __forceinline__ void halo_cell(const Geom &g, const TileGeom &t, const Lay<TWC> &l,
                                          const TileOrigin &o, int n, int &cell, int64_t &gi,
                                          bool &in, int &kind) {
    const int TW = tile_w<TWC>(t);
    const int ncol = 2 * t.TH * g.K;
    int yl, j, wl;
    if (n < ncol) {
        kind = n & 1;
        j = t.rTH ? (int)__umulhi((unsigned)(n >> 1), t.rTH) : n >> 1;
        yl = (n >> 1) - j * t.TH;
        wl = kind ? TW : -1;
    } else {
        n -= ncol;
        j = n / TW;
        wl = n - j * TW;
        kind = 2;
        yl = -1;
        if (j >= g.K) {
            j -= g.K;
            kind = 3;
            yl = t.TH;
        }
    }
    const int W = o.W0 + wl, y = o.y0 + yl;
    cell = l.cell(yl, j, wl);
    in = W >= 0 && W < g.ng && y >= 0 && y < g.h;
    gi = ((int64_t)y * g.K + j) * g.P + W;
}

// Loads of a halo cell: the height, and the residual words stored at the head
// of an arc of the tile's own nodes (rr, ri1 left; ri0 right; rd, ri3 top; ri2
// bottom).  Positions outside the grid get height kInfH and zero residuals.
__device__ __forceinline__ void halo_load(const SolveArgs &a, const int32_t *hsrc, bool with_res,
                                          int64_t gi, bool in, int kind, int32_t &h, int32_t &r1,
                                          int32_t &r2) {
    const State &s = a.s;
    h = (in && hsrc) ? ld(&hsrc[gi]) : kInfH;   // hsrc NULL: heights unknown (infinite)
    r1 = r2 = 0;
    if (with_res && in) {
        if (kind == 0) {
            r1 = ld(&s.rr[gi]);
            r2 = ld(&s.ri1[gi]);
        } else if (kind == 1) {
            r1 = ld(&s.ri0[gi]);
        } else if (kind == 2) {
            r1 = ld(&s.rd[gi]);
            r2 = ld(&s.ri3[gi]);
        } else {
            r1 = ld(&s.ri2[gi]);
        }
    }
}

// Fields of a halo cell that hold the words of arcs from the tile's own nodes
// (by kind, -1: none), the arrays they come from, and two fields it does not
// use, where a sweep visit keeps the words as loaded.  Its excess field adds
// up the flow a sweep visit pushes into it, from 1: a halo node always looks as
// if it had excess before a push, so it never joins the visit's active nodes.
__device__ __forceinline__ int halo_f1(int kind) {
    return kind == 0 ? F_RR : kind == 1 ? F_I0 : kind == 2 ? F_RD : F_I2;
}
__device__ __forceinline__ int halo_f2(int kind) { return kind == 0 ? F_I1 : kind == 2 ? F_I3 : -1; }
enum { F_KEEP1 = F_RC, F_KEEP2_COL = F_RD, F_KEEP2_ROW = F_RR };
__device__ __forceinline__ int halo_k2(int kind) { return kind == 0 ? F_KEEP2_COL : F_KEEP2_ROW; }

template <int TWC>
__device__ __forceinline__ void halo_store(int32_t *sm, const Lay<TWC> &l, bool with_res, int cell,
                                           int kind, int32_t h, int32_t r1, int32_t r2) {
    int32_t *c = sm + cell;
    c[l.at(F_HT)] = h;
    if (!with_res) return;
    c[l.at(F_EX)] = 1;
    c[l.at(halo_f1(kind))] = r1;
    c[l.at(F_KEEP1)] = r1;
    if (halo_f2(kind) >= 0) {
        c[l.at(halo_f2(kind))] = r2;
        c[l.at(halo_k2(kind))] = r2;
    }
}

template <int TWC>
__device__ __forceinline__ int halo_cells(const Geom &g, const TileGeom &t) {
    return 2 * g.K * (t.TH + tile_w<TWC>(t));
}

template <int TWC>
__device__ __forceinline__ void halo_issue(const SolveArgs &a, const Lay<TWC> &l,
                                           const TileOrigin &o, bool with_res,
                                           const int32_t *hsrc, HaloRegs &hr) {
    const int total = halo_cells<TWC>(a.g, a.t);
#pragma unroll
    for (int u = 0; u < 2; u++) {
        const int n = threadIdx.x + u * blockDim.x;
        hr.cell[u] = 0;
        hr.kind[u] = -1;
        hr.h[u] = kInfH;
        hr.r1[u] = hr.r2[u] = 0;
        if (n >= total) continue;
        int64_t gi;
        bool in;
        halo_cell<TWC>(a.g, a.t, l, o, n, hr.cell[u], gi, in, hr.kind[u]);
        halo_load(a, hsrc, with_res, gi, in, hr.kind[u], hr.h[u], hr.r1[u], hr.r2[u]);
    }
}

template <int TWC>
__device__ __forceinline__ void halo_commit(int32_t *sm, const Lay<TWC> &l, bool with_res,
                                            const HaloRegs &hr) {
#pragma unroll
    for (int u = 0; u < 2; u++)
        if (hr.kind[u] >= 0)
            halo_store<TWC>(sm, l, with_res, hr.cell[u], hr.kind[u], hr.h[u], hr.r1[u], hr.r2[u]);
}

template <int TWC>
__device__ __forceinline__ void halo_rest(const SolveArgs &a, int32_t *sm, const Lay<TWC> &l, const TileOrigin &o,
                          bool with_res, const int32_t *hsrc) {
    const int total = halo_cells<TWC>(a.g, a.t);
    for (int n = threadIdx.x + 2 * blockDim.x; n < total; n += blockDim.x) {
        int cell, kind;
        int64_t gi;
        bool in;
        halo_cell<TWC>(a.g, a.t, l, o, n, cell, gi, in, kind);
        int32_t h, r1, r2;
        halo_load(a, hsrc, with_res, gi, in, kind, h, r1, r2);
        halo_store<TWC>(sm, l, with_res, cell, kind, h, r1, r2);
    }
}

// A thread's block of own nodes: its site, first layer and number of layers
// (0: the thread has no such block).
struct Own {
    int wl, yl, j0, n;
};

template <int TWC>
__device__ __forceinline__ Own own_block(const Geom &g, const TileGeom &t, int u) {
    const int id = threadIdx.x + u * blockDim.x;
    const int blk = (int)__umulhi((unsigned)id, t.rS), site = id - blk * t.S;
    const int TW = tile_w<TWC>(t);
    Own w;
    w.yl = site / TW;
    w.wl = site - w.yl * TW;
    w.j0 = blk * kBlk;
    w.n = min(kBlk, max(0, g.K - w.j0));
    return w;
}

// Search direction of a relabel pass (see SolveArgs::dir).
__device__ __forceinline__ int eff_dir(const SolveArgs &a) {
    if (a.dir != 2) return a.dir;
    return ld(&a.s.hdr->rev) ? 0 : 1;
}

// ---------------------------------------------------------- relabel pass ---

// Local relaxation to the tile's fixed point.  Own nodes' residual-arc masks
// are in registers (mk), own heights and halo heights in shared memory.

// One word per block of layers at the end of the tile's shared memory, that of
// block b at b + 1 (the outer two stay 0): how often a height of the block of
// any site changed.  Cleared before the staging barrier of a relabel visit.
__device__ __forceinline__ uint32_t *block_words(int32_t *sm, const TileGeom &t) {
    return (uint32_t *)sm + t.words;
}
__device__ __forceinline__ void clear_blocks(int32_t *sm, const TileGeom &t) {
    uint32_t *w = block_words(sm, t);
    for (int b = threadIdx.x; b < t.nblk + 2; b += blockDim.x) w[b] = 0;
}

// Heights of a block from those around it: a lateral minimum per node, then
// one pass up and one pass down the block, which is exact along the chain.
// 30 loads for four nodes instead of 14 each, and a height crosses a block of
// the chain in one step: with one node per thread a tile of 63 layers took as
// many dependent steps as the chain has layers (16 us a visit).  Returns
// whether a height changed.
template <int TWC>
__device__ __forceinline__ bool relax_block(const Lay<TWC> &l, volatile int32_t *c, int n,
                                            const unsigned (&mk)[kBlk]) {
    const volatile int32_t *up = c - l.sy, *dn = c + l.sy;
    int32_t h[kBlk], b[kBlk], L[kBlk + 2], R[kBlk + 2], U[kBlk + 2], D[kBlk + 2];
#pragma unroll
    for (int k = 0; k < kBlk; k++) h[k] = c[l.at(F_HT, k)];
    const int32_t hb = c[l.at(F_HT, -1)], ha = c[l.at(F_HT, kBlk)];
#pragma unroll
    for (int k = 0; k < kBlk + 2; k++) {
        L[k] = c[l.at(F_HT, k - 1, -1)];
        R[k] = c[l.at(F_HT, k - 1, 1)];
        U[k] = up[l.at(F_HT, k - 1)];
        D[k] = dn[l.at(F_HT, k - 1)];
    }
#pragma unroll
    for (int k = 0; k < kBlk; k++) {
        const unsigned m = mk[k];
        int32_t x = kInfH, y = kInfH;
        if (m & (1u << 2)) x = min(x, R[k + 1]);
        if (m & (1u << 3)) y = min(y, L[k + 1]);
        if (m & (1u << 4)) x = min(x, D[k + 1]);
        if (m & (1u << 5)) y = min(y, U[k + 1]);
        if (m & (1u << 6)) x = min(x, L[k]);
        if (m & (1u << 7)) y = min(y, R[k]);
        if (m & (1u << 8)) x = min(x, U[k]);
        if (m & (1u << 9)) y = min(y, D[k]);
        if (m & (1u << 10)) x = min(x, L[k + 2]);
        if (m & (1u << 11)) y = min(y, R[k + 2]);
        if (m & (1u << 12)) x = min(x, U[k + 2]);
        if (m & (1u << 13)) y = min(y, D[k + 2]);
        if (k >= n) h[k] = kInfH;                 // past the chain's end
        b[k] = min(h[k], min(x, y) + 1);
    }
#pragma unroll
    for (int k = 0; k < kBlk; k++)
        if (mk[k] & 2u) b[k] = min(b[k], (k ? b[k - 1] : hb) + 1);
#pragma unroll
    for (int k = kBlk - 1; k >= 0; k--)
        if (mk[k] & 1u) b[k] = min(b[k], (k < kBlk - 1 ? b[k + 1] : ha) + 1);
    bool ch = false;
#pragma unroll
    for (int k = 0; k < kBlk; k++) {
        if (b[k] < h[k] && k < n) {
            c[l.at(F_HT, k)] = b[k];
            ch = true;
        }
    }
    return ch;
}

template <int TPT, int TWC>
__device__ __forceinline__ bool relax_tile(const SolveArgs &a, int32_t *sm, const int (&cell)[TPT],
                           const int (&nl)[TPT], const unsigned (&mk)[TPT][kBlk],
                           int max_outer = 1 << 30, const unsigned *done_ctr = nullptr,
                           unsigned items = 0, bool *cut = nullptr) {
    const TileGeom &t = a.t;
    const Lay<TWC> l(t);
    // Asynchronous (chaotic) relaxation: each warp relaxes its blocks, reading
    // neighbours' heights as other warps update them.  Values only decrease
    // and stay upper bounds, so any interleaving converges to the same fixed
    // point.
    // A block's heights depend on its own and the two adjacent blocks of
    // layers, so a warp leaves its blocks alone unless one of these changed
    // since it last looked (block_words): the fronts of a relaxation touch a
    // few layers at a time.  A round ends at a barrier; one in which no height
    // changed anywhere proves that the fixed point has been reached.  (Up to
    // eight sweeps of a warp between barriers took 8 % longer: most warps
    // wait for the one that goes on.)
    const int lane = threadIdx.x & 31;
    volatile uint32_t *chg = block_words(sm, t);
    const bool uniform = (t.S & 31) == 0;        // a warp's blocks lie in one row of blocks
    // lanes 16 u + i watch the i-th of the blocks around this warp's blocks u
    // (at most 8 + 2 of them); the others watch block -1, which never changes
    int watch = 0;
    int blk[TPT];
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        const int id0 = (threadIdx.x & ~31) + u * blockDim.x;
        const int lo = (int)__umulhi((unsigned)id0, t.rS);
        const int hi = min((int)__umulhi((unsigned)(id0 + 31), t.rS), t.nblk - 1);
        blk[u] = (int)__umulhi((unsigned)(id0 + lane), t.rS);
        const int i = lane - 16 * u;
        if (i >= 0 && i < 16 && lo < t.nblk && i < hi - lo + 3) watch = lo + i;
    }
    uint32_t last = 0;
    bool any_change = false;
    // Straggler cut (with done_ctr): after a round that changed heights, stop
    // when all but 1 + min(items / 8, half the grid) of the step's items are
    // done (the last items of a step much larger than the grid are not
    // stragglers: they started late).  The caller queues the tile again, and
    // the heights so far are upper bounds of the fixed point, so a later pass
    // resumes from them.  Thread 0 loads the done count every other round and
    // looks at it two rounds later (a round is shorter than the load), and
    // publishes its decision before the round's barrier, in a slot the next
    // round does not overwrite.
    __shared__ int s_rstop[2];
    const unsigned margin = 1 + min(items / 8, gridDim.x / 2);
    unsigned seen = 0;
    int stop = 0;
    for (int outer = 0;; outer++) {
        int changed = 0;
        if (done_ctr && threadIdx.x == 0 && (outer & 1) == 0) {
            stop = outer >= 2 && seen + margin >= items;
            seen = *(volatile const unsigned *)done_ctr;
        }
        // A warp that has seen a count must see the heights it counts, or it
        // would rest on old ones after the barrier too: the count is read before
        // the heights, and a writer's heights are visible before it counts them,
        // with a fence on either side (the warp barriers carry it to all lanes).
        const uint32_t now = chg[watch];
        const bool fresh = __any_sync(0xffffffffu, now != last);
        last = now;
        if (fresh || outer == 0) {
            __threadfence_block();
            __syncwarp();
#pragma unroll
            for (int u = 0; u < TPT; u++) {
                const bool ch = cell[u] > 0 && relax_block<TWC>(l, sm + cell[u], nl[u], mk[u]);
                if (__any_sync(0xffffffffu, ch)) {
                    changed = 1;
                    __syncwarp();
                    if (uniform ? lane == 0 : ch) {
                        __threadfence_block();
                        red_add_smem((int32_t *)&chg[blk[u] + 1], 1);
                    }
                }
            }
        }
        if (done_ctr && threadIdx.x == 0) s_rstop[outer & 1] = stop;
        if (!__syncthreads_or(changed)) break;
        any_change = true;
        if (outer + 1 >= max_outer) break;
        if (done_ctr && s_rstop[outer & 1]) {
            *cut = true;
            break;
        }
    }
    return any_change;
}

// Active count of a relabel visit and the neighbour sides it changed, zeroed
// before the visit's staging barrier.
__shared__ int s_count;
__shared__ unsigned s_sides;

// First relabel pass of a tile: residual-arc masks from the current state,
// heights reset (0 on nodes with sink capacity left, else infinity), local
// relaxation with an unknown (infinite) halo.  Returns the tile's active
// count (positive excess and a finite height).
template <int TPT, int TWC, class Halfway>
__device__ __forceinline__ int relabel_init_tile(const SolveArgs &a, int32_t *sm, int tile,
                                                 Halfway halfway) {
    const Geom &g = a.g;
    const TileGeom &t = a.t;
    const State &s = a.s;
    const Lay<TWC> l(t);
    const TileOrigin o = tile_origin(t, tile);
    const int dir = eff_dir(a);
    // halo heights are not known yet in this pass: staged as infinite
    HaloRegs hr;
    halo_issue<TWC>(a, l, o, true, nullptr, hr);
    clear_blocks(sm, t);
    if (threadIdx.x == 0) s_count = 0;
    int cell[TPT], nl[TPT];      // cell > 0: a block of the grid
    unsigned mk[TPT][kBlk];
    int64_t gi[TPT];
    int32_t v_rc[TPT][kBlk], v_rr[TPT][kBlk], v_rd[TPT][kBlk], v_r0[TPT][kBlk], v_r1[TPT][kBlk],
        v_r2[TPT][kBlk], v_r3[TPT][kBlk], v_ex[TPT][kBlk];
    // own nodes: every load first ...
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        const Own w = own_block<TWC>(g, t, u);
        const int W = o.W0 + w.wl, y = o.y0 + w.yl;
        nl[u] = w.n;
        cell[u] = w.n ? l.cell(w.yl, w.j0, w.wl) : 0;
        if (W >= g.ng || y >= g.h) cell[u] = -cell[u];
        gi[u] = ((int64_t)y * g.K + w.j0) * g.P + W;
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            mk[u][k] = 0;
            v_rc[u][k] = v_rr[u][k] = v_rd[u][k] = v_r0[u][k] = v_r1[u][k] = v_r2[u][k] =
                v_r3[u][k] = v_ex[u][k] = 0;
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int64_t i = gi[u] + (int64_t)k * g.P;
            v_rc[u][k] = ld(&s.rc[i]);
            v_rr[u][k] = ld(&s.rr[i]);
            v_rd[u][k] = ld(&s.rd[i]);
            v_r0[u][k] = ld(&s.ri0[i]);
            v_r1[u][k] = ld(&s.ri1[i]);
            v_r2[u][k] = ld(&s.ri2[i]);
            v_r3[u][k] = ld(&s.ri3[i]);
            v_ex[u][k] = ld(&s.ex[i]);
        }
    }
    // ... then the shared-memory stores
    halo_commit<TWC>(sm, l, true, hr);
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        int32_t *c = sm + abs(cell[u]);
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (cell[u] == 0 || k >= nl[u]) continue;
            if (cell[u] < 0) {
                c[l.at(F_HT, k)] = kInfH;
                continue;
            }
            c[l.at(F_RC, k)] = v_rc[u][k];
            c[l.at(F_RR, k)] = v_rr[u][k];
            c[l.at(F_RD, k)] = v_rd[u][k];
            c[l.at(F_I0, k)] = v_r0[u][k];
            c[l.at(F_I1, k)] = v_r1[u][k];
            c[l.at(F_I2, k)] = v_r2[u][k];
            c[l.at(F_I3, k)] = v_r3[u][k];
            const int32_t e = v_ex[u][k];
            c[l.at(F_HT, k)] = (dir == 0 ? e < 0 : e > 0) ? 0 : kInfH;
        }
    }
    halo_rest<TWC>(a, sm, l, o, true, nullptr);
    __syncthreads();
    halfway();
#pragma unroll
    for (int u = 0; u < TPT; u++) {
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int32_t *c = sm + cell[u] + l.at(0, k);
            int32_t r[kSlots];
            load_residuals<TWC>(l, g, c, r);
            unsigned m = 0;
            if (dir == 0) {
                // arc u -> head
#pragma unroll
                for (int q = 0; q < kSlots; q++) m |= r[q] > 0 ? 1u << q : 0u;
            } else {
                // arc head -> u: the reverse of the data arc up is infinite, that
                // of the one down is the data arc of layer j - 1, else the
                // pair's rest
                m = 1u | (c[l.at(F_RC, -1)] > 0 ? 2u : 0u);
#pragma unroll
                for (int q = 2; q < kSlots; q++) {
                    const int32_t cap = q < 6 ? g.lam2 : q == 8 || q == 9 || q >= 12 ? g.h2v : g.h2h;
                    m |= cap - r[q] > 0 ? 1u << q : 0u;
                }
            }
            mk[u][k] = m | (dir == 0 && v_ex[u][k] > 0 ? 0x8000u : 0u);
            __stcg(&a.amask[gi[u] + (int64_t)k * g.P], (uint16_t)mk[u][k]);
        }
    }
    // (no barrier: the masks read words that only the staging wrote)
    // the first pass's relaxation is capped: the pass after it visits every
    // tile again, with the halo known, and relaxes each to its fixed point
    relax_tile<TPT, TWC>(a, sm, cell, nl, mk, kInitOuter);
    int act = 0;
#pragma unroll
    for (int u = 0; u < TPT; u++) {
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int32_t h = sm[cell[u] + l.at(F_HT, k)];
            __stcg(&a.hgt[gi[u] + (int64_t)k * g.P], h);
            act += (mk[u][k] & 0x8000u) && h < kInfH;
        }
    }
    act = __reduce_add_sync(0xffffffffu, act);
    if ((threadIdx.x & 31) == 0 && act) atomicAdd(&s_count, act);
    __syncthreads();
    if (threadIdx.x == 0) __stcg(&a.tile_cnt[tile], s_count);
    return s_count;
}

// Queue a tile for the next step, once: the caller that turns its flag from 0
// to 1 appends it to the list, and the tile's visit in that step clears the
// flag again.
__device__ __forceinline__ void enqueue(int32_t *flag, int32_t *list, int32_t *count, int tile) {
    if (atomicExch(&flag[tile], 1) == 0) __stcg(&list[atomicAdd(count, 1)], tile);
}

// Neighbour tile on side q (0: W-1, 1: W+1, 2: y-1, 3: y+1), or -1.
__device__ __forceinline__ int side_tile(const TileGeom &t, const TileOrigin &o, int tile, int q) {
    if (q == 0) return o.tx > 0 ? tile - 1 : -1;
    if (q == 1) return o.tx + 1 < t.tiles_w ? tile + 1 : -1;
    if (q == 2) return o.ty > 0 ? tile - t.tiles_w : -1;
    return o.ty + 1 < t.tiles_h ? tile + t.tiles_w : -1;
}

// Later relabel passes: masks from the first pass, heights from global
// memory (own and halo); relax, write back what changed, mark the neighbour
// tiles whose halo changed, and return the change of the tile's active count
// (the marks are warp 0's and come after the visit's last block barrier).
template <int TPT, int TWC, class Halfway>
__device__ __forceinline__ int relabel_pass_tile(const SolveArgs &a, int32_t *sm, int tile, int &changed,
                                 int32_t *dirty_next, int32_t *list_next, int32_t *count_next,
                                 const unsigned *done_ctr, unsigned items, Halfway halfway) {
    const Geom &g = a.g;
    const TileGeom &t = a.t;
    const Lay<TWC> l(t);
    const TileOrigin o = tile_origin(t, tile);
    const int before = ld(&a.tile_cnt[tile]);    // issued now, used at the end
    HaloRegs hr;
    halo_issue<TWC>(a, l, o, false, a.hgt, hr);
    clear_blocks(sm, t);
    if (threadIdx.x == 0) {
        s_count = 0;
        s_sides = 0;
    }
    int cell[TPT], nl[TPT];      // cell > 0: a block of the grid
    unsigned mk[TPT][kBlk];
    int64_t gi[TPT];
    int32_t h0[TPT][kBlk];
    // own nodes: every load first, then the shared-memory stores
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        const Own w = own_block<TWC>(g, t, u);
        const int W = o.W0 + w.wl, y = o.y0 + w.yl;
        nl[u] = w.n;
        cell[u] = w.n ? l.cell(w.yl, w.j0, w.wl) : 0;
        if (W >= g.ng || y >= g.h) cell[u] = -cell[u];
        gi[u] = ((int64_t)y * g.K + w.j0) * g.P + W;
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            mk[u][k] = 0;
            h0[u][k] = kInfH;
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int64_t i = gi[u] + (int64_t)k * g.P;
            mk[u][k] = ld(&a.amask[i]);
            h0[u][k] = ld(&a.hgt[i]);
        }
    }
    halo_commit<TWC>(sm, l, false, hr);
#pragma unroll
    for (int u = 0; u < TPT; u++)
#pragma unroll
        for (int k = 0; k < kBlk; k++)
            if (cell[u] && k < nl[u]) sm[abs(cell[u]) + l.at(F_HT, k)] = h0[u][k];
    halo_rest<TWC>(a, sm, l, o, false, a.hgt);
    __syncthreads();
    halfway();
    bool cut = false;
    const bool ch = relax_tile<TPT, TWC>(a, sm, cell, nl, mk, 1 << 30, done_ctr, items, &cut);
    int act = 0;
    unsigned sides = 0;
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        bool moved = false;
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int32_t h = sm[cell[u] + l.at(F_HT, k)];
            if (h != h0[u][k]) {
                __stcg(&a.hgt[gi[u] + (int64_t)k * g.P], h);
                moved = true;
            }
            act += (mk[u][k] & 0x8000u) && h < kInfH;
        }
        if (moved) {
            const Own w = own_block<TWC>(g, t, u);
            sides |= (w.wl == 0 ? 1u : 0u) | (w.wl == tile_w<TWC>(t) - 1 ? 2u : 0u) |
                     (w.yl == 0 ? 4u : 0u) | (w.yl == t.TH - 1 ? 8u : 0u);
        }
    }
    act = __reduce_add_sync(0xffffffffu, act);
    sides = __reduce_or_sync(0xffffffffu, sides);
    if ((threadIdx.x & 31) == 0) {
        if (act) atomicAdd(&s_count, act);
        if (sides) atomicOr(&s_sides, sides);
    }
    __syncthreads();
    if (threadIdx.x < 4 && (s_sides >> threadIdx.x & 1u)) {
        const int nb = side_tile(t, o, tile, threadIdx.x);
        if (nb >= 0) enqueue(dirty_next, list_next, count_next, nb);
    }
    // a relaxation cut short goes on in the next pass
    if (cut && threadIdx.x == 4) enqueue(dirty_next, list_next, count_next, tile);
    if (ch) changed = 1;
    if (threadIdx.x == 0) __stcg(&a.tile_cnt[tile], s_count);
    return s_count - before;
}

// ------------------------------------------------------------ sweep visit ---

// One arc slot of a tile shape; in a sweep visit a lane holds four.  Offsets
// count from the node's cell, in bytes.
//   .x  shared offset of the residual word
//   .y  shared offset of the head's cell
//   .z, .w  residual = z + w * word: 0, 1 when the word is stored at the node (a push
//       subtracts); the pair's capacity, -1 when it is stored at the head (a push adds);
//       infinite, 0 for the reverse data arc (a push adds to the head's word)
// Entries 14 and 15 are no arcs: the node itself, never residual.
__shared__ int4 s_slot[16];

__device__ __forceinline__ int4 make_slot(const Geom &g, const TileGeom &t, int q) {
    // head (dy, dj, dw) and field of the word
    static constexpr int8_t tab[kSlots][4] = {
        {0, 1, 0, F_RC},  {0, -1, 0, F_RC},  {0, 0, 1, F_RR},  {0, 0, -1, F_RR}, {1, 0, 0, F_RD},
        {-1, 0, 0, F_RD}, {0, -1, -1, F_I0}, {0, -1, 1, F_I1}, {-1, -1, 0, F_I2}, {1, -1, 0, F_I3},
        {0, 1, -1, F_I1}, {0, 1, 1, F_I0},   {-1, 1, 0, F_I3}, {1, 1, 0, F_I2}};
    if (q >= kSlots) return make_int4(0, 0, 0, 0);
    const int off = tab[q][0] * t.SYs + tab[q][1] * F_N * t.SJ + tab[q][2];
    const bool at_head = q == 3 || q == 5 || q >= 10;
    const int cap = q < 6 ? g.lam2 : q < 12 ? g.h2h : g.h2v;
    return make_int4(4 * (tab[q][3] * t.SJ + (at_head || q == 1 ? off : 0)), 4 * off,
                     q == 1 ? kInfR : at_head ? cap : 0, q == 1 ? 0 : at_head ? -1 : 1);
}

// Fill the block's tables for the tile shape of pair a: s_slot, and the
// padding between the rows of a tile.
__device__ void build_tables(const SolveArgs &a, int32_t *sm) {
    const Geom &g = a.g;
    const TileGeom &t = a.t;
    if (threadIdx.x < 16) s_slot[threadIdx.x] = make_slot(g, t, threadIdx.x);
    const int layer = F_N * t.SJ, pad = t.SYs - (g.K + 1) * layer;
    for (int r = 0; r <= t.TH + 2; r++) {
        const int to = min(t.words, r * t.SYs + layer);
        for (int w = max(0, r * t.SYs - pad) + threadIdx.x; w < to; w += blockDim.x) sm[w] = kInfH;
    }
}

// Lists of a sweep visit's active nodes (positive excess, finite height), as
// cells, for the iteration running and the next: two halves of TN entries
// behind the block words, and one entry more that takes what goes nowhere.
// Their lengths, by iteration mod kLens (warp 0 may run half as many ahead).
constexpr int kLens = 64;
__shared__ int s_nodes[kLens];

// Discharge the eight nodes of a list (shared address `list`, n entries) from
// entry `first` on, four lanes to a node: lane q of the four holds arc slots
// 4 q .. 4 q + 3 (st), the last one also the node's own words.  A lane loads
// its arcs' residuals and its heads' heights, a saturating scan over the four
// lanes deals the excess out to the admissible slots in slot order (chain arcs
// first; another order took 20 % more visits), and each lane pushes its
// share; a minimum over the same lanes gives the relabel.  Flow into the halo
// gathers in the halo cells' excess and words.
// A node joins the next list when a push takes its excess above zero, or when
// it has excess left after its own discharge: once in either case.
// A warp is bound by the chain of dependent instructions here, and an
// iteration has 17 to 45 active nodes on average: one lane per node ran the
// code of 14 slots for lanes most of which were idle, and sixteen or eight
// lanes per node took as long for two or four nodes as four lanes do for eight.
template <int TWC>
__device__ __forceinline__ void discharge(const Lay<TWC> &l, unsigned base, unsigned list,
                                          int first, int n, const int4 (&st)[4], unsigned next,
                                          unsigned next_n, unsigned nowhere) {
    const int lane = threadIdx.x & 31, q = lane & 3;
    const int i = first + (lane >> 2);
    unsigned c;
    asm volatile("{ .reg .u16 h; ld.volatile.shared.u16 h, [%1]; cvt.u32.u16 %0, h; }"
                 : "=r"(c) : "r"(list + 2 * min(i, n - 1)));
    c = base + 4 * c;
    int32_t e = lds(c + 4 * l.at(F_EX));
    const int32_t hu = lds(c + 4 * l.at(F_HT));
    int32_t w[4], hv[4], x[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        w[j] = lds(c + st[j].x);
        hv[j] = lds(c + st[j].y + 4 * l.at(F_HT));
    }
    if (i >= n) e = 0;
    int32_t hm = kInfH;
    unsigned sum = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int32_t r = (int32_t)((unsigned)st[j].z + (unsigned)st[j].w * (unsigned)w[j]);
        // (a head that does not exist has an infinite height)
        x[j] = r > 0 && hv[j] < hu ? min(r, e) : 0;
        hm = min(hm, r > 0 && hv[j] >= hu ? hv[j] : kInfH);
        sum = min(sum + (unsigned)x[j], (unsigned)e);
    }
#pragma unroll
    for (int s = 1; s < 4; s <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, sum, s, 4);
        hm = min(hm, __shfl_xor_sync(0xffffffffu, hm, s));
        if (q >= s) sum = min(sum + y, (unsigned)e);
    }
    const unsigned y = __shfl_up_sync(0xffffffffu, sum, 1, 4);
    const bool own = q == 3;
    const int32_t tot = (int32_t)sum;            // lane 3: all the flow pushed
    int32_t left = e - (q ? (int32_t)y : 0), old[4];
    unsigned ea[4];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        x[j] = min(x[j], left);
        left -= x[j];
        ea[j] = c + st[j].y + 4 * l.at(F_EX);
        // (the arc's word needs no atomic: in one iteration only one of its ends
        // can push along it -- each would have to lie above the other, and
        // heights only rise)
        old[j] = push_words(c + st[j].x, st[j].w > 0 ? w[j] - x[j] : w[j] + x[j], x[j], ea[j],
                            j == 2 && own ? -tot : x[j]);
    }
    // lane 3: every admissible slot is saturated: relabel over the others
    const bool stuck = own && tot < e;
    const int32_t h = !stuck ? hu : hm >= kInfH - 1 ? kInfH : hm + 1;
    sts(stuck ? c + 4 * l.at(F_HT) : nowhere, h);
    bool join[4];
    int joins = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        join[j] = x[j] > 0 && old[j] <= 0 && old[j] + x[j] > 0;
        if (j == 2 && own) join[j] = (tot ? old[j] - tot : e) > 0 && h < kInfH;
        joins += join[j];
    }
    unsigned at = next + 2 * (unsigned)atom_add_nz(next_n, joins);
#pragma unroll
    for (int j = 0; j < 4; j++) {
        sts16(join[j] ? at : nowhere, (int)((ea[j] - base) >> 2));
        if (join[j]) at += 2;
    }
}

// Up to `iters` push/relabel iterations of one tile in shared memory.  (The
// visit ends with a block barrier.)
template <int TPT, int TWC, class Halfway>
__device__ __forceinline__ void sweep_tile(const SolveArgs &a, int32_t *sm, int tile, int round, int iters,
                           int &overflow, int32_t *list_next, int32_t *count_next,
                           const unsigned *done_ctr, unsigned items, Halfway halfway) {
    const Geom &g = a.g;
    const TileGeom &t = a.t;
    const State &s = a.s;
    const Lay<TWC> l(t);
    const TileOrigin o = tile_origin(t, tile);
    int32_t *act_next = a.tile_act + ((round + 1) & 1) * t.T;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5, W = blockDim.x >> 5;
    __shared__ unsigned s_touch;
    __shared__ int s_stop[2];        // in turn: written before an iteration's barrier
    __shared__ int s_it;
    if (threadIdx.x == 0) s_touch = 0;   // read only after the staging barrier below
    if (threadIdx.x < kLens) s_nodes[threadIdx.x] = 0;
    HaloRegs hr;
    halo_issue<TWC>(a, l, o, true, s.ht, hr);
    int cell[TPT], nl[TPT];      // cell > 0: a block of the grid
    int64_t gi[TPT];
    int32_t o_ex[TPT][kBlk], o_rc[TPT][kBlk], o_rr[TPT][kBlk], o_rd[TPT][kBlk], o_r0[TPT][kBlk],
        o_r1[TPT][kBlk], o_r2[TPT][kBlk], o_r3[TPT][kBlk], o_ht[TPT][kBlk];
    // own nodes: every load first (the originals stay in registers for the
    // write-back as deltas) ...
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        const Own w = own_block<TWC>(g, t, u);
        const int Wg = o.W0 + w.wl, y = o.y0 + w.yl;
        nl[u] = w.n;
        cell[u] = w.n ? l.cell(w.yl, w.j0, w.wl) : 0;
        if (Wg >= g.ng || y >= g.h) cell[u] = -cell[u];
        gi[u] = ((int64_t)y * g.K + w.j0) * g.P + Wg;
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            o_ex[u][k] = o_rc[u][k] = o_rr[u][k] = o_rd[u][k] = o_r0[u][k] = o_r1[u][k] =
                o_r2[u][k] = o_r3[u][k] = 0;
            o_ht[u][k] = kInfH;
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int64_t i = gi[u] + (int64_t)k * g.P;
            o_ex[u][k] = ld(&s.ex[i]);
            o_ht[u][k] = ld(&s.ht[i]);
            o_rc[u][k] = ld(&s.rc[i]);
            o_rr[u][k] = ld(&s.rr[i]);
            o_rd[u][k] = ld(&s.rd[i]);
            o_r0[u][k] = ld(&s.ri0[i]);
            o_r1[u][k] = ld(&s.ri1[i]);
            o_r2[u][k] = ld(&s.ri2[i]);
            o_r3[u][k] = ld(&s.ri3[i]);
        }
    }
    // ... then the shared-memory stores
    halo_commit<TWC>(sm, l, true, hr);
#pragma unroll
    for (int u = 0; u < TPT; u++) {
        int32_t *c = sm + abs(cell[u]);
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (cell[u] == 0 || k >= nl[u]) continue;
            c[l.at(F_EX, k)] = o_ex[u][k];
            c[l.at(F_HT, k)] = o_ht[u][k];
            if (cell[u] < 0) continue;
            c[l.at(F_RC, k)] = o_rc[u][k];
            c[l.at(F_RR, k)] = o_rr[u][k];
            c[l.at(F_RD, k)] = o_rd[u][k];
            c[l.at(F_I0, k)] = o_r0[u][k];
            c[l.at(F_I1, k)] = o_r1[u][k];
            c[l.at(F_I2, k)] = o_r2[u][k];
            c[l.at(F_I3, k)] = o_r3[u][k];
        }
    }
    halo_rest<TWC>(a, sm, l, o, true, s.ht);
    __syncthreads();
    halfway();
    // the first list
    const unsigned base = (unsigned)__cvta_generic_to_shared(sm);
    const unsigned lists = base + 4 * (t.words + t.nblk + 2), nowhere = lists + 4 * t.TN;
    {
        unsigned b[TPT][kBlk];
        int total = 0;
#pragma unroll
        for (int u = 0; u < TPT; u++)
#pragma unroll
            for (int k = 0; k < kBlk; k++) {
                b[u][k] = __ballot_sync(0xffffffffu, o_ex[u][k] > 0 && o_ht[u][k] < kInfH);
                total += __popc(b[u][k]);
            }
        int at = 0;
        if (lane == 0 && total) at = atomicAdd(&s_nodes[0], total);
        at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
        for (int u = 0; u < TPT; u++)
#pragma unroll
            for (int k = 0; k < kBlk; k++) {
                const int i = at + __popc(b[u][k] & ((1u << lane) - 1u));
                sts16((b[u][k] >> lane) & 1u ? lists + 2 * i : nowhere, cell[u] + l.at(F_EX, k));
                at += __popc(b[u][k]);
            }
    }
    const int4 st[4] = {s_slot[4 * (lane & 3)], s_slot[4 * (lane & 3) + 1],
                        s_slot[4 * (lane & 3) + 2], s_slot[4 * (lane & 3) + 3]};
    // Local iterations: the warps share out the nodes of the list, and the
    // iteration ends with a block barrier.  (With a list of its own per warp
    // and no barrier, the last warp took twice the average.)  While the list
    // is one discharge's worth, warp 0 goes on by itself, without barriers
    // (40 % of the iterations).  Discharges run concurrently on shared memory;
    // the lock-free argument that holds between tiles holds between warps
    // (only a node's own discharge lowers its excess, and residuals are
    // consumed only by an arc's tail).
    // Straggler cut: a step ends when its last item does, so a visit still
    // running when nearly all of its step's items are done (all but 1 +
    // min(items / 8, half the grid)) stops after half its local iterations.
    // Its tile keeps its work and is queued for the next round.  Thread 0
    // loads the step's done count every fourth iteration and looks at it two
    // iterations later (an iteration is shorter than the load).  No cut
    // without done_ctr (fixed-sweep mode: a round is a full round).
    const unsigned margin = 1 + min(items / 8, gridDim.x / 2);
    const unsigned counts = (unsigned)__cvta_generic_to_shared(s_nodes);
    unsigned seen = 0;
    bool stop = false, shared = false;
    int it = 0, turn = 0;
    auto iteration = [&](int i, int first, int n) {
        if (threadIdx.x == 0) {
            if (done_ctr && (i & 3) == 0) seen = *(volatile const unsigned *)done_ctr;
            if (done_ctr && (i & 3) == 2) stop = seen + margin >= items;
            s_nodes[(i + kLens / 2) % kLens] = 0;
        }
#pragma unroll 1
        for (; first < n; first += 8 * W)
            discharge<TWC>(l, base, lists + 2 * t.TN * (i & 1), first, n, st,
                           lists + 2 * t.TN * ((i + 1) & 1), counts + 4 * ((i + 1) % kLens),
                           nowhere);
    };
    __syncthreads();
    while (it < iters) {
        int n = s_nodes[it % kLens];
        if (n == 0) break;
        if (n > 8 || shared) {
            iteration(it, 8 * warp, n);
            if (threadIdx.x == 0) s_stop[turn] = stop;
            __syncthreads();
            it++;
            if (it >= iters / 2 && s_stop[turn]) break;
            turn ^= 1;
            shared = false;
        } else {
            if (warp == 0) {
                int i = it, cut = 0;
                do {
                    iteration(i, 0, n);
                    __syncwarp();
                    n = *(volatile int *)&s_nodes[++i % kLens];
                    if (i >= iters / 2 && __shfl_sync(0xffffffffu, (int)stop, 0)) {
                        cut = 1 << 30;
                        break;
                    }
                } while (i < iters && n > 0 && n <= 8 && i - it < kLens / 2 - 4);
                if (lane == 0) s_it = i | cut;
            }
            __syncthreads();
            it = s_it & ~(1 << 30);
            if (s_it != it) break;
            shared = true;       // (s_it is read before the next barrier)
        }
    }
    // active nodes are left when the list of the next iteration has entries
    const bool left = s_nodes[it % kLens] != 0;
    // flow pushed into halo nodes: their excess, and the words stored at them
    unsigned bits = left ? 16u : 0u;
    const int cells = halo_cells<TWC>(g, t);
    for (int n = threadIdx.x; n < cells; n += blockDim.x) {
        int hc, kind;
        int64_t gh;
        bool in;
        halo_cell<TWC>(g, t, l, o, n, hc, gh, in, kind);
        const int32_t *c = sm + hc;
        const int32_t v = c[l.at(F_EX)] - 1;
        if (v == 0) continue;
        red_add_gmem(&s.ex[gh], v);
        bits |= 1u << kind;
        const int64_t gs = s.rr - s.rc;          // global fields are equally spaced
        int32_t d = c[l.at(halo_f1(kind))] - c[l.at(F_KEEP1)];
        if (d) red_add_gmem(s.rc + (halo_f1(kind) - F_RC) * gs + gh, d);
        if (halo_f2(kind) >= 0) {
            d = c[l.at(halo_f2(kind))] - c[l.at(halo_k2(kind))];
            if (d) red_add_gmem(s.rc + (halo_f2(kind) - F_RC) * gs + gh, d);
        }
    }
    // one barrier for the tile's flags: bits 0-3 neighbour tiles that received
    // flow (left, right, up, down), bit 4 work left in this tile, bit 5 overflow
    bits = __reduce_or_sync(0xffffffffu, bits);
    if (lane == 0 && bits) atomicOr(&s_touch, bits);
    __syncthreads();
    // The last warp queues the tiles with work while it writes its own nodes
    // back: two round trips to L2, that of the flag and that of the place in
    // the list, which took 1.2 of a visit's 16 us when they came after the
    // write-back (19 sizes: 2.4 % less in the mean, 349x338x42 7 %).
    int to = -1, was = 1, at = 0;
    const bool queue = warp == W - 1 && lane < 5 && (s_touch >> lane & 1u);
    if (queue) {
        to = lane == 4 ? tile : side_tile(t, o, tile, lane);
        if (to >= 0) was = atomicExch(&act_next[to], 1);
    }
    // write back own nodes as deltas (other tiles may have updated the same
    // words through global atomics meanwhile)
    bool over = false;
#pragma unroll
    for (int u = 0; u < TPT; u++) {
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (queue && u == 0 && k == 2 && was == 0) at = atomicAdd(count_next, 1);
            if (cell[u] <= 0 || k >= nl[u]) continue;
            const int32_t *c = sm + cell[u] + l.at(0, k);
            const int64_t i = gi[u] + (int64_t)k * g.P;
            const int32_t ex = c[l.at(F_EX)], ht = c[l.at(F_HT)], rc = c[l.at(F_RC)];
            // the data-arc residual is the one word that can grow without a
            // bound of its own (flow pushed back down the infinite reverse
            // arc); only this tile changes it (the chain stays inside the tile)
            over |= rc > kCapLimit || rc < 0;
            red_add_nz(&s.ex[i], ex - o_ex[u][k]);
            red_add_nz(&s.rc[i], rc - o_rc[u][k]);
            red_add_nz(&s.rr[i], c[l.at(F_RR)] - o_rr[u][k]);
            red_add_nz(&s.rd[i], c[l.at(F_RD)] - o_rd[u][k]);
            red_add_nz(&s.ri0[i], c[l.at(F_I0)] - o_r0[u][k]);
            red_add_nz(&s.ri1[i], c[l.at(F_I1)] - o_r1[u][k]);
            red_add_nz(&s.ri2[i], c[l.at(F_I2)] - o_r2[u][k]);
            red_add_nz(&s.ri3[i], c[l.at(F_I3)] - o_r3[u][k]);
            stg_if(ht != o_ht[u][k], &s.ht[i], ht);
        }
    }
    if (queue && was == 0) __stcg(&list_next[at], to);
    if (__any_sync(0xffffffffu, over) && lane == 0) atomicOr(&s_touch, 32u);
    __syncthreads();
    overflow = (s_touch & 32u) != 0;
}

// ------------------------------------------------------- the solve loop ---
//
// One cooperative launch solves n independent pairs.  Each pair runs its own
// sequence of steps; in a step each of its tiles with work does the pair's
// current phase:
//
//   INIT   first relabel pass (masks, heights reset, in-tile distances)
//   PASS   later relabel pass (all tiles once, then tiles whose halo changed)
//   SWEEP  one sweep round over the tiles with work
//   LABELS label extraction (extraction launches)
//   DONE   nothing
//
// A step's work items are all T tiles of the pair (INIT, the first PASS, the
// first SWEEP round -- those with active nodes -- and LABELS) or the tiles
// queued for it by the visits of the step before.  Blocks claim items one at
// a time from a per-pair claim word (step | items | next item), taking them
// from any pair that has some; the block that completes a step's last item
// advances that pair's state machine and publishes its next step.  There is
// no grid barrier: a pair in a latency-bound tail steps as fast as its own
// visits allow while other blocks work on other pairs.
// Per pair the schedule is the one of a single solve: a relabel (capped at
// relabel_passes passes unless it decides termination), then sweep rounds --
// sweeps_per_relabel of them, or in the tail (few active nodes) until the
// tiles with work stop decreasing and the sweep rounds have cost as much as the
// relabel did, both counted in tile visits one CTA makes in sequence.

constexpr int kMaxPairs = 64;
enum { PH_INIT = 0, PH_PASS = 1, PH_SWEEP = 2, PH_LABELS = 3, PH_DONE = 4 };

struct PairState {
    int phase, pass, full, conv, tail, status, cap;
    int exact_end;     // ended on a relabel run to its fixed point that found nothing active
    int ht_labels;     // extraction reads the solve's exact heights (no relabel of its own)
    long long round, nrounds, rounds_total, relabels, passes, outer;
    long long active, prev1, prev2, relabel_visits, relabel_depth, last_relabel_depth, sweep_depth;
    long long visits_sweep_total, visits_relabel_total;
    long long ns_sweep, ns_relabel;    // device time of the steps in each phase
    unsigned long long t_step;         // start of the current step (global timer)
};

// Per-pair control words of a launch.  claim packs the current step's queue
// slot (step mod 3), its number of items and the next item (24 bits each):
// one atomic add both claims an item and tells where its step's queue is.
// The words that idle blocks poll (claim), that running visits poll (done),
// that visits add to, and the state lie in cache lines of their own.
struct PairCtl {
    alignas(128) unsigned long long claim;
    alignas(128) unsigned int done;   // items of the current step completed
    alignas(128) long long red[3][4]; // per-step sums (slot = step mod 3)
    int32_t qcount[3];                // queued tiles per step slot
    unsigned int step;                // current step
    alignas(128) PairState st;        // written only by the block that advances the pair
};

constexpr unsigned kItemMask = 0xffffffu;
// An idle block gives up after this long unless the options set a limit.
constexpr unsigned long long kDefaultIdleLimitNs = 60ull * 1000 * 1000 * 1000;

constexpr int kStateWords = sizeof(PairState) / 8;
static_assert(sizeof(PairState) % 8 == 0 && kStateWords <= 28, "a warp copies PairState, a word a lane");

// Copy of a pair's state as other SMs wrote it (L2-coherent loads).
__device__ __forceinline__ void load_state(PairState *dst, const PairState *src) {
    const long long *s = (const long long *)src;
    long long *d = (long long *)dst;
    for (int i = 0; i < (int)(sizeof(PairState) / 8); i++) d[i] = __ldcg(s + i);
}

__device__ __forceinline__ unsigned long long pack_claim(unsigned step, unsigned items,
                                                         unsigned next) {
    // bits 48-63: the step's queue slot (step mod 3), so a block that claims
    // an item knows where the step's queue is from the claim alone
    return ((unsigned long long)(step % 3u) << 48) |
           ((unsigned long long)(items & kItemMask) << 24) | (next & kItemMask);
}

struct BatchArgs {
    int n;            // pairs
    int extract;      // 0: max-flow solve, 1: label extraction
    unsigned long long idle_limit_ns;   // a block idle this long aborts the launch
    Ctrl *bar;        // abort flag and the count of finished pairs (Ctrl::active)
    PairCtl *ctl;     // [n]
    SolveArgs pair[kMaxPairs];
};

static_assert(sizeof(BatchArgs) <= 32000, "the batch arguments travel as kernel parameters");

__device__ void start_relabel(PairState &st, const SolveArgs &a) {
    if (a.mode == GS_MODE_EXACT && st.outer >= a.max_iters) {
        st.phase = PH_DONE;
        st.status = GS_ERR_TIMEOUT;
        return;
    }
    st.outer++;
    st.phase = PH_INIT;
    st.relabel_visits = 0;
    st.relabel_depth = 0;
}

// Critical-path cost of a step that visited `visits` tiles of a pair: the
// number of tile visits one CTA makes in sequence, at least one.
__device__ __forceinline__ long long step_depth(long long visits) {
    return max(1ll, (visits + gridDim.x - 1) / gridDim.x);
}

// Advance one pair at the end of a step; v = the step's sums {a, b, c, overflow}.
__device__ void advance(PairState &st, const SolveArgs &a, const long long v[4], int extract) {
    if (v[3] && st.status == GS_OK) {
        st.status = GS_ERR_OVERFLOW;
        st.phase = PH_DONE;
        return;
    }
    switch (st.phase) {
        case PH_INIT:
            st.active = v[0];
            st.relabel_visits = v[2];
            st.relabel_depth = step_depth(v[2]);
            st.passes++;
            st.pass = 1;
            st.phase = PH_PASS;
            break;
        case PH_PASS: {
            st.active += v[0];
            st.relabel_visits += v[2];
            st.relabel_depth += step_depth(v[2]);
            st.passes++;
            bool end = false;
            st.conv = 0;
            if (v[1] == 0) {
                st.conv = 1;
                end = true;
            } else if (!extract && !st.full && st.pass >= st.cap) {
                end = true;
            } else {
                st.pass++;
            }
            if (!end) break;
            if (extract) {
                st.phase = PH_LABELS;
                break;
            }
            st.relabels++;
            st.last_relabel_depth = st.relabel_depth;
            // a relabel run to its fixed point because the capped one reached no
            // active node, and that found some: later relabels reach as far
            if (st.full && st.active > 0) st.cap = max(st.cap, st.pass);
            st.visits_relabel_total += st.relabel_visits;
            if (st.active == 0) {
                if (st.conv) {
                    st.phase = PH_DONE;
                    st.exact_end = 1;
                } else {
                    st.full = 1;     // nothing active within reach: decide with an exact relabel
                    start_relabel(st, a);
                }
                break;
            }
            st.full = 0;
            st.tail = st.active * 64 <= (long long)a.g.N;
            st.nrounds = st.tail ? 64ll * a.sweeps_per_relabel : a.sweeps_per_relabel;
            if (a.mode == GS_MODE_FIXED_SWEEPS) {
                st.nrounds = min(st.nrounds, a.fixed_sweeps - st.rounds_total);
                if (st.nrounds <= 0) {
                    st.phase = PH_DONE;
                    break;
                }
            }
            st.round = 0;
            st.sweep_depth = 0;
            st.prev1 = st.prev2 = 1ll << 40;
            st.phase = PH_SWEEP;
            break;
        }
        case PH_SWEEP: {
            const long long worked = v[0];
            st.rounds_total++;
            st.round++;
            st.sweep_depth += step_depth(worked);
            st.visits_sweep_total += worked;
            const bool stalled = st.tail && st.round >= 3 && worked * 10 > st.prev2 * 9 &&
                                 st.sweep_depth > st.last_relabel_depth;
            st.prev2 = st.prev1;
            st.prev1 = worked;
            if (worked == 0 || stalled || st.round >= st.nrounds) {
                if (a.mode == GS_MODE_FIXED_SWEEPS && st.rounds_total >= a.fixed_sweeps)
                    st.phase = PH_DONE;
                else
                    start_relabel(st, a);
            }
            break;
        }
        case PH_LABELS:
            st.active = v[0];      // sink capacity left
            if (v[1]) st.status = GS_ERR_LABELS;
            st.phase = PH_DONE;
            break;
        default:
            break;
    }
}

// Labels of one tile's sites and the tile's remaining sink capacity.  A thread
// counts the source-side nodes of its blocks of layers; the source side of a
// chain must be a prefix, so a source-side node lies above another or is the
// first.  (One thread per site walked the whole chain with the other threads
// idle: 1.85 ms for 514x480 sites of 63 layers.)
__device__ long long labels_tile(const SolveArgs &a, int32_t *sm, int tile, const int32_t *hsrc,
                                 int &bad) {
    const Geom &g = a.g;
    const TileGeom &t = a.t;
    const TileOrigin o = tile_origin(t, tile);
    int32_t *count = sm + t.words + t.nblk + 2;      // [S], where sweeps keep their lists
    unsigned long long deficit = 0;
    int b = 0;
    const int dir = eff_dir(a);
    const bool rev = ld(&a.s.hdr->rev) != 0;
    for (int site = threadIdx.x; site < t.S; site += blockDim.x) count[site] = 0;
    __syncthreads();
    for (int u = 0; u < a.tpt; u++) {
        const Own w = own_block<0>(g, t, u);
        const int W = o.W0 + w.wl, y = o.y0 + w.yl;
        if (!w.n || W >= g.ng || y >= g.h) continue;
        const int64_t i = ((int64_t)y * g.K + w.j0) * g.P + W;
        int32_t h[kBlk + 1], e[kBlk];
#pragma unroll
        for (int k = 0; k <= kBlk; k++)              // h[0]: the layer below the block
            h[k] = k <= w.n && w.j0 + k > 0 ? ld(&hsrc[i + (int64_t)(k - 1) * g.P]) : 0;
#pragma unroll
        for (int k = 0; k < kBlk; k++) e[k] = k < w.n ? ld(&a.s.ex[i + (int64_t)k * g.P]) : 0;
        auto in = [&](int32_t v) { return dir == 1 ? v < kInfH : v >= kInfH; };
        bool prev = w.j0 == 0 || in(h[0]);
        int n = 0;
#pragma unroll
        for (int k = 0; k < kBlk; k++) {
            if (k >= w.n) break;
            const bool now = in(h[k + 1]);
            b |= now && !prev;
            n += now;
            prev = now;
            if (e[k] < 0) deficit += (unsigned long long)(-(int64_t)e[k]);
        }
        if (n) atomicAdd(&count[w.yl * t.TW + w.wl], n);
    }
    __syncthreads();
    for (int site = threadIdx.x; site < t.S; site += blockDim.x) {
        const int yl = site / t.TW, W = o.W0 + site - yl * t.TW, y = o.y0 + yl;
        if (W < g.ng && y < g.h)
            a.labels[(int64_t)y * g.ng + W] = rev ? g.D - 1 - count[site] : count[site];
    }
    bad = __syncthreads_or(b);
    return block_sum((long long)deficit);
}

// Phases whose items are the tiles queued by the step before.
__device__ __forceinline__ bool queued(const PairState &st) {
    return (st.phase == PH_PASS && st.pass > 1) || (st.phase == PH_SWEEP && st.round > 0);
}

// Items of a pair's step from its state and the queue the step before filled.
__device__ __forceinline__ unsigned step_items(const PairState &st, const SolveArgs &a,
                                               const PairCtl *c, unsigned step) {
    if (st.phase == PH_DONE) return 0;
    return queued(st) ? (unsigned)*(volatile const int32_t *)&c->qcount[step % 3] : (unsigned)a.t.T;
}

// Statistics and results of a finished pair.
__device__ void pair_results(const BatchArgs &B, const PairState &st, const SolveArgs &a,
                             int status) {
    if (!B.extract) {
        Ctrl *c = a.ctrl;
        c->stats[0] = st.relabels;
        c->stats[1] = st.rounds_total;
        c->stats[2] = st.passes;
        c->stats[4] = st.active;
        c->stats[5] = st.ns_sweep;
        c->stats[6] = st.ns_relabel;
        c->stats[7] = 1;
        c->visits_sweep = st.visits_sweep_total;
        c->visits_relabel = st.visits_relabel_total;
        c->converged = st.phase == PH_DONE && status == GS_OK;
        // the heights are then the exact distances to the remaining sink
        // capacity: an extraction that needs just those reuses them
        if (st.exact_end && status == GS_OK) a.s.hdr->exact_heights = 1;
    } else {
        a.ctrl->stats[3] = st.passes;
        *a.flow = (int64_t)a.s.hdr->init_deficit - st.active;
    }
    if (status != GS_OK) atomicCAS(a.status, GS_OK, status);
}

// End of a pair's step (one warp, after every item completed): advance the
// state machine -- through any steps that have no items -- and publish the
// next step's claim word, or count the pair finished.  s_st holds the pair's
// state, unchanged since the step began.
__device__ __forceinline__ void end_step(const BatchArgs &B, int p, int slot, PairState &s_st) {
    PairCtl *c = B.ctl + p;
    const SolveArgs &a = B.pair[p];
    const int lane = threadIdx.x & 31;
    // the step's sums, the queue the step filled for the next one and its
    // number, loaded together (the caller's acquire on the done count orders
    // them after every item's writes)
    long long mine = 0;
    if (lane < 4) mine = *(volatile long long *)&c->red[slot][lane];
    else if (lane == 4) mine = *(volatile int32_t *)&c->qcount[(slot + 1) % 3];
    else if (lane == 5) mine = *(volatile unsigned *)&c->step;
    long long v0[4];
#pragma unroll
    for (int k = 0; k < 4; k++) v0[k] = __shfl_sync(0xffffffffu, mine, k);
    const int32_t q0 = (int32_t)__shfl_sync(0xffffffffu, mine, 4);
    unsigned step = (unsigned)__shfl_sync(0xffffffffu, mine, 5);
    unsigned items = 0;
    bool finished = false;
    if (lane == 0) {
        PairState st = s_st;
        bool first = true;
        const unsigned long long t_now = now_ns();
        if (st.phase == PH_SWEEP) st.ns_sweep += (long long)(t_now - st.t_step);
        else st.ns_relabel += (long long)(t_now - st.t_step);
        st.t_step = t_now;
        for (;;) {
            long long v[4];
            const bool pre = first && step % 3 == (unsigned)slot;   // the prefetched words apply
            if (pre)
                for (int k = 0; k < 4; k++) v[k] = v0[k];
            else
                for (int k = 0; k < 4; k++) v[k] = *(volatile long long *)&c->red[step % 3][k];
            first = false;
            advance(st, a, v, B.extract);
            const unsigned next = step + 1;
            for (int k = 0; k < 4; k++) c->red[next % 3][k] = 0;
            c->qcount[(next + 1) % 3] = 0;
            items = st.phase == PH_DONE ? 0u
                    : (pre && queued(st)) ? (unsigned)q0
                                          : step_items(st, a, c, next);
            step = next;
            if (st.phase == PH_DONE || items > 0) break;
        }
        c->done = 0;
        c->step = step;
        s_st = st;
        finished = st.phase == PH_DONE;
        if (finished) pair_results(B, st, a, st.status);
    }
    __syncwarp();
    if (lane < kStateWords) ((long long *)&c->st)[lane] = ((const long long *)&s_st)[lane];
    __syncwarp();
    if (lane == 0) {
        atom_exch_release(&c->claim, pack_claim(step, items, 0));
        if (finished) atomicAdd(&B.bar->active, 1);
    }
}

// The item a block works on.
struct Item {
    int p, tile, slot;      // pair, tile, queue slot of the step (tile < 0: the launch is over)
    unsigned items, idx;    // items of the step, this one's number
};

// The block's next item of the same step, claimed while it works on this one
// (thread 0): the claim's result, then the tile it names.  Only while the step
// has two items or more left for every block, so that its end stays shared out.
struct Ahead {
    unsigned long long w;
    int32_t tile, count;    // queued tile (or the item's number); its active nodes
    int abort;
    bool has;
};

// Halfway through a visit (thread 0): look up the item claimed ahead.
__device__ __forceinline__ void look_ahead(const BatchArgs &B, const SolveArgs &a, const Item &it,
                                           bool queued, Ahead &ah) {
    if (threadIdx.x != 0 || !ah.has) return;
    const unsigned idx = (unsigned)(ah.w & kItemMask);
    ah.has = idx < it.items;
    if (!ah.has) return;
    ah.tile = queued ? ld(&a.tile_list[it.slot * a.t.T + idx]) : (int)idx;
    ah.count = ld(&a.tile_cnt[idx]);
    ah.abort = *(volatile int32_t *)&B.bar->abort;
}

// Sums of a completed item (active nodes or worked tiles, changes, visits, overflow).
struct ItemSums {
    long long a, b, c;
    int ovf;
};

// Complete the block's item `it` (it.tile >= 0: a visit with sums v) and claim
// the next one that has work, into it and s_st (warp 0; the caller's block
// barrier hands them to the other warps).
// The atomic that claims the next item of the same step goes out before the
// one that counts the completed item, so the two round trips overlap; the
// words a claimed item needs are loaded by one lane each.
// With an item claimed ahead there is nothing to wait for: this one cannot be
// the step's last, so it is counted without looking at the count, and the
// pair's state is the same.
__device__ __forceinline__ void next_item(const BatchArgs &B, Item &it, const ItemSums &v0,
                                          const Ahead &ah, PairState &s_st) {
    const int lane = threadIdx.x & 31;
    ItemSums v = v0;
    bool finish = it.tile >= 0;
    if (__shfl_sync(0xffffffffu, (int)ah.has, 0)) {
        if (lane == 0) {
            PairCtl *c = B.ctl + it.p;
            long long *rp = c->red[it.slot];
            if (v.a) atomicAdd((unsigned long long *)&rp[0], (unsigned long long)v.a);
            if (v.b) atomicAdd((unsigned long long *)&rp[1], (unsigned long long)v.b);
            if (v.c) atomicAdd((unsigned long long *)&rp[2], (unsigned long long)v.c);
            if (v.ovf) atomicAdd((unsigned long long *)&rp[3], 1ull);
            red_add_release(&c->done, 1u);
        }
        it.idx = (unsigned)(__shfl_sync(0xffffffffu, ah.w, 0) & kItemMask);
        it.tile = __shfl_sync(0xffffffffu, ah.tile, 0);
        if (__shfl_sync(0xffffffffu, ah.abort, 0)) it.tile = -1;
        if (it.tile < 0 || queued(s_st) || s_st.phase != PH_SWEEP ||
            __shfl_sync(0xffffffffu, ah.count, 0) > 0)
            return;
        v.a = v.b = v.c = 0;             // nothing to sweep in that tile
        v.ovf = 0;
    }
    for (;;) {
        unsigned long long w = 0;
        bool got = false;
        if (finish) {
            PairCtl *c = B.ctl + it.p;
            // (only with more items left than blocks: near the end of a step
            // its completion must not wait for a claim that may find nothing)
            const bool more = it.idx + gridDim.x < it.items;
            bool last = false;
            if (lane == 0) {
                long long *rp = c->red[it.slot];
                if (v.a) atomicAdd((unsigned long long *)&rp[0], (unsigned long long)v.a);
                if (v.b) atomicAdd((unsigned long long *)&rp[1], (unsigned long long)v.b);
                if (v.c) atomicAdd((unsigned long long *)&rp[2], (unsigned long long)v.c);
                if (v.ovf) atomicAdd((unsigned long long *)&rp[3], 1ull);
                if (more) w = atom_add_relaxed(&c->claim, 1ull);
                // a release (the item's writes before it) and an acquire (every
                // item's writes, and what the claim above names, after it); the
                // step cannot end before this item does
                last = atom_add_acq_rel(&c->done, 1u) + 1u == it.items;
            }
            w = __shfl_sync(0xffffffffu, w, 0);
            if (__shfl_sync(0xffffffffu, (int)last, 0)) end_step(B, it.p, it.slot, s_st);
            got = more && (w & kItemMask) < ((w >> 24) & kItemMask);
        }
        int p = it.p, over = 0;
        if (!got && lane == 0) {
            // poll the pairs' claim words; idle polling backs off to 256 ns
            const unsigned long long t0 = now_ns();
            for (int spin = 0; !got && !over; spin++) {
                if (aborted(B.bar) || *(volatile int32_t *)&B.bar->active >= B.n) {
                    over = 1;
                    break;
                }
                for (int k = 0; k < B.n && !got; k++) {
                    p = (int)((blockIdx.x + k) % B.n);
                    PairCtl *c = B.ctl + p;
                    w = *(volatile unsigned long long *)&c->claim;
                    if ((w & kItemMask) >= ((w >> 24) & kItemMask)) continue;
                    w = atom_add_acquire(&c->claim, 1ull);
                    got = (w & kItemMask) < ((w >> 24) & kItemMask);
                }
                if (got) break;
                if (now_ns() - t0 > B.idle_limit_ns) {
                    atomicExch(&B.bar->abort, 1);
                    over = 1;
                    break;
                }
                __nanosleep(32u << min(spin, 3));
            }
        }
        p = __shfl_sync(0xffffffffu, p, 0);
        w = __shfl_sync(0xffffffffu, w, 0);
        it.tile = -1;
        if (__shfl_sync(0xffffffffu, over, 0)) return;
        it.p = p;
        it.slot = (int)((w >> 48) & 3u);
        it.items = (unsigned)((w >> 24) & kItemMask);
        it.idx = (unsigned)(w & kItemMask);
        // everything the item needs, loaded together: the pair's state, both
        // ways the item may name its tile (the queued tile at this slot, or
        // tile idx with its count of active nodes), and the abort flag
        const SolveArgs &a = B.pair[p];
        const PairCtl *c = B.ctl + p;
        int32_t x = 0;
        if (lane < kStateWords)
            ((long long *)&s_st)[lane] = __ldcg((const long long *)&c->st + lane);
        else if (lane == 29) x = ld(&a.tile_list[it.slot * a.t.T + it.idx]);
        else if (lane == 30) x = ld(&a.tile_cnt[it.idx]);
        else if (lane == 31) x = *(volatile int32_t *)&B.bar->abort;
        __syncwarp();
        const int qt = __shfl_sync(0xffffffffu, x, 29), tc = __shfl_sync(0xffffffffu, x, 30);
        if (__shfl_sync(0xffffffffu, x, 31)) return;      // aborted: leave (tile stays -1)
        it.tile = queued(s_st) ? qt : (int)it.idx;
        if (queued(s_st) || s_st.phase != PH_SWEEP || tc > 0) return;
        // nothing to sweep in this tile: complete at once
        v.a = v.b = v.c = 0;
        v.ovf = 0;
        finish = true;
    }
}

// One item of a step.
struct Visit {
    int tile, next, T;
    unsigned items;
    const BatchArgs &B;
    const Item &it;
};

template <int TPT, int TWC>
__device__ __forceinline__ void visit_tile(const SolveArgs &a, PairCtl *c, const PairState &st,
                                           const Visit &v, int32_t *sm, ItemSums &sums,
                                           Ahead &ah) {
    // between a visit's staging and its work, when the claim ahead is back
    auto halfway = [&]() { look_ahead(v.B, a, v.it, queued(st), ah); };
    int32_t *list_next = a.tile_list + v.next * v.T;
    int32_t *count_next = &c->qcount[v.next];
    const int tile = v.tile;
    if (st.phase == PH_INIT) {
        if (threadIdx.x == 0) {
            __stcg(&a.tile_dirty[tile], 0);
            __stcg(&a.tile_dirty[v.T + tile], 0);
            __stcg(&a.tile_act[tile], 0);
            __stcg(&a.tile_act[v.T + tile], 0);
        }
        sums.a = relabel_init_tile<TPT, TWC>(a, sm, tile, halfway);
        sums.c = 1;
    } else if (st.phase == PH_PASS) {
        const int pass = st.pass;
        int32_t *dcur = a.tile_dirty + (pass & 1) * v.T;
        int32_t *dnext = a.tile_dirty + ((pass + 1) & 1) * v.T;
        if (pass > 1 && threadIdx.x == 0) __stcg(&dcur[tile], 0);
        int ch = 0;
        sums.a = relabel_pass_tile<TPT, TWC>(a, sm, tile, ch, dnext, list_next, count_next, &c->done,
                                             v.items, halfway);
        sums.b = ch;
        sums.c = 1;
    } else {   // PH_SWEEP
        const int cur = (int)(st.round & 1);
        if (threadIdx.x == 0) __stcg(&a.tile_act[cur * v.T + tile], 0);
        const int iters = st.tail ? a.tail_iters : a.local_iters;
        const unsigned *done_ctr = a.mode == GS_MODE_FIXED_SWEEPS ? nullptr : &c->done;
        sweep_tile<TPT, TWC>(a, sm, tile, cur, iters, sums.ovf, list_next, count_next, done_ctr,
                             v.items, halfway);
        sums.a = 1;
    }
}

// What bounds a launch: the chain of dependent instructions of its tile visits
// (a fifth to a quarter of the issue slots are used, DRAM at a few percent) and,
// where a step has few items, the wait for its last one (62 % of the block time
// at 384x288x16, 10 % at 640x480x64) with a hand-over of about 4 us.  Visits in
// us as staging + work + write-back, measured in a copy with counters, with a
// node per lane and a warp's own lists -> as it is:
//   384x288x16 (8x8 tiles, 2 x 256 threads an SM): sweep 2.7 + 11.7 + 2.8 -> 2.5 +
//     9.1 + 2.5, relabel 1.3 + 4.3 + 1.7 -> 1.0 + 3.1 + 1.0, first pass 5.8 + 5.2 + 0.5
//     -> 2.7 + 4.6 + 0.4; the solve 13.1 -> 10.6 ms
//   640x480x64 (8x4, 512 threads): sweep 4.7 + 8.7 + 2.6 -> 3.9 + 9.8 + 2.7 for a third
//     fewer visits, relabel 2.1 + 16.0 + 1.9 -> 1.6 + 4.9 + 1.1, first pass 8.2 + 5.8 +
//     0.4 -> 4.4 + 4.5 + 0.3; the solve 225 -> 106 ms
// An iteration takes 0.72 us for up to 64 nodes in 512 threads (0.66 by one warp).
// A warp's discharge is 0.45 us of it: loads 97 cycles, admissibility and scan 230,
// pushes 290, the place in the next list 230, the entries' stores 82.  The other
// 0.27 us are the loop, the list's length and the barrier with the wait for the
// slowest warp.
// Registers: one block of nodes per thread takes all 128 and spills 32 bytes; two
// (explicit shapes only, and every pair of a batch that holds one) spill 884, and
// still take half the time of the node-per-lane code on the same shapes
// (500x400x48, 8x8: 43 against 84 ms).
//
// TPT: blocks of own nodes per thread, the most any pair of the launch needs.
// Blocks of 256 or 512 threads; 128 registers a thread leave room for two or
// one of them per SM.
template <int TPT>
__global__ void __launch_bounds__(kTileThreads, 1) k_batch(const __grid_constant__ BatchArgs B) {
    extern __shared__ int32_t smem[];
    __shared__ Item s_item;
    __shared__ PairState s_st;
    int tables_for = -1;           // pair whose tile-shape tables the block holds
    // block 0 starts every pair and publishes its first step
    if (blockIdx.x == 0) {
        for (int p = threadIdx.x; p < B.n; p += blockDim.x) {
            PairCtl *c = B.ctl + p;
            PairState st;
            memset(&st, 0, sizeof(st));
            st.status = GS_OK;
            st.cap = B.pair[p].relabel_passes;
            st.t_step = now_ns();
            const SolveArgs &a = B.pair[p];
            if (!B.extract) {
                a.s.hdr->exact_heights = 0;
                start_relabel(st, a);
            } else if (a.dir == 2 && ld(&a.s.hdr->rev) && ld(&a.s.hdr->exact_heights)) {
                // the label-reversed problem's labels come from distances to the
                // sink capacity, which the finished solve left exact in ht
                st.phase = PH_LABELS;
                st.ht_labels = 1;
            } else {
                start_relabel(st, a);
            }
            c->st = st;
            c->step = 0;
            c->done = 0;
            const unsigned items = step_items(st, B.pair[p], c, 0);
            if (st.phase == PH_DONE) pair_results(B, st, B.pair[p], st.status);
            __threadfence();
            atomicExch(&c->claim, pack_claim(0, items, 0));
            if (st.phase == PH_DONE) atomicAdd(&B.bar->active, 1);
        }
    }
    Item it = {0, -1, 0, 0, 0};
    ItemSums sums = {0, 0, 0, 0};
    Ahead ah = {0, 0, 0, 0, false};
    for (;;) {
        if (threadIdx.x < 32) {
            next_item(B, it, sums, ah, s_st);
            if (threadIdx.x == 0) s_item = it;
        }
        __syncthreads();
        it = s_item;
        if (it.tile < 0) break;
        PairCtl *c = B.ctl + it.p;
        const SolveArgs &a = B.pair[it.p];
        if (it.p != tables_for) {    // uniform: every thread read the same item
            build_tables(a, smem);
            tables_for = it.p;
            __syncthreads();
        }
        sums = {0, 0, 0, 0};
        ah.has = threadIdx.x == 0 && it.idx + 2 * gridDim.x < it.items;
        if (ah.has) ah.w = atom_add_relaxed(&c->claim, 1ull);
        // (a visit has a block barrier after its last look at s_item and s_st; a
        // relabel visit ends with warp 0's queueing)
        if (s_st.phase != PH_LABELS) {
            // the visit's code for this tile width, and a pair whose tiles
            // need one block per thread runs that code also when the launch is
            // sized for two
            const Visit v = {it.tile, (it.slot + 1) % 3, a.t.T, it.items, B, it};
            if (TPT == 2 && a.tpt == 1) {
                if (a.t.TW == 8) visit_tile<1, 8>(a, c, s_st, v, smem, sums, ah);
                else if (a.t.TW == 16) visit_tile<1, 16>(a, c, s_st, v, smem, sums, ah);
                else visit_tile<1, 0>(a, c, s_st, v, smem, sums, ah);
            } else {
                if (a.t.TW == 8) visit_tile<TPT, 8>(a, c, s_st, v, smem, sums, ah);
                else if (a.t.TW == 16) visit_tile<TPT, 16>(a, c, s_st, v, smem, sums, ah);
                else visit_tile<TPT, 0>(a, c, s_st, v, smem, sums, ah);
            }
        } else {
            int bad = 0;
            look_ahead(B, a, it, false, ah);
            sums.a = labels_tile(a, smem, it.tile, s_st.ht_labels ? a.s.ht : a.hgt, bad);
            sums.b = bad;
        }
        __syncwarp();
    }
    // pairs still running when the launch gave up
    if (blockIdx.x == 0 && aborted(B.bar)) {
        __syncthreads();
        for (int p = threadIdx.x; p < B.n; p += blockDim.x) {
            PairState st;
            load_state(&st, &B.ctl[p].st);
            if (st.phase != PH_DONE) pair_results(B, st, B.pair[p], GS_ERR_TIMEOUT);
        }
    }
}

// ------------------------------------------------------------ host side ---

// Shared-memory conflicts of the first warp's lanes (their blocks' cells) for a
// row stride: the largest number of lanes on one bank.
static int bank_conflicts(int TW, int S, int SJ, int sy) {
    int hits[32] = {}, worst = 0;
    for (int n = 0; n < 32; n++) {
        const int site = n % S;
        const int w = (site / TW) * sy + (n / S) * kBlk * 9 * SJ + site % TW;
        worst = std::max(worst, ++hits[w & 31]);
    }
    return worst;
}

// Bytes of a tile's nine fields over its nodes and a one-site halo, rows padded
// to TW (mod 32) where a warp takes whole rows: the size that the shape rules
// (and gs_tile_info) go by.  0: never a tile.
static size_t field_bytes(const Geom &g, int TW, int TH, int bt) {
    const int64_t TN = (int64_t)TH * g.K * TW;
    if (TN > 8 * bt || TN > 4096 || g.K >= 2048) return 0;
    int row = g.K * (TW + 2);
    if (TH % (32 / TW) == 0) row += ((TW - row) % 32 + 32) % 32;
    const int64_t cells = (int64_t)(TH + 2) * row;
    return cells < 8192 ? 9 * cells * sizeof(int32_t) : 0;
}

// Tile shape: whole chains (all K layers), TW sites x TH rows, the nine fields
// within 180 KB; one block of kBlk layers per thread, or two.  The library's
// own choice prefers one, and with 256-thread blocks fields within 80 KB, so
// that two tiles fit an SM (long chains fall back to one).  The kernel takes more
// shared memory than the fields (a layer of padding between rows of sites, the
// lists of active nodes): 216124 bytes for 184320 at the most, a third more at
// 9 depth numbers, 3.4 times as much at 2, where the padding is as large as the
// chains.  `fields` returns field_bytes of the shape, `smem` what the kernel
// needs, within a block's 227 KB.
static bool pick_tile(const Geom &g, TileGeom &t, int &tpt, size_t &smem, int want_w = 0,
                      int want_h = 0, int bt = kTileThreads, size_t *fields = nullptr) {
    const size_t budgets[2] = {(bt == 256 && !want_w ? 80 : 180) * size_t(1024), 180 * 1024};
    // More sites first, squarer first among equals: a breadth-first path then
    // crosses fewer tile borders, and a visit's fixed cost (staging, claims,
    // write-back: half of it) is spread over more sites.  With the number of
    // blocks of layers between two powers of two only rows of 5, 6 or 7 sites
    // fill the threads.  500x300 pairs, 512 threads, ms: 20 depth numbers 8x8
    // 22.0, 16x6 18.3; 36: 8x4 39.3, 8x7 29.2; 44: 8x4 42.2, 8x5 36.9; 700x400x40:
    // 8x4 93.8, 8x6 68.4, and 8x8 with two blocks per thread 79.5 (its visits
    // spill); 32: 8x8 24.7, 8x7 26.1.  16x5 against 8x8 gains on no side: 24 depth
    // numbers, 200x200 13.2 and 12.0, 600x400 42.6 and 42.7.
    static const int cand[][2] = {{16, 8}, {16, 6}, {8, 8}, {16, 4}, {32, 4}, {8, 7}, {8, 6},
                                  {8, 5},  {8, 4},  {32, 2}, {16, 2}, {4, 8}, {8, 3}, {8, 2},
                                  {4, 4},  {16, 1}, {8, 1},  {4, 2},  {4, 1}};
    if (want_w || want_h) {
        if (!(want_w == 4 || want_w == 8 || want_w == 16 || want_w == 32) || want_h < 1 ||
            want_h > 8)
            return false;
    }
    for (int pass = 0; pass < 4; pass++) {
        for (int ci = 0; ci < (want_w ? 1 : (int)(sizeof(cand) / sizeof(cand[0]))); ci++) {
            const int TW = want_w ? want_w : cand[ci][0], TH = want_w ? want_h : cand[ci][1];
            const size_t fb = field_bytes(g, TW, TH, bt);
            if (!fb || fb > budgets[pass / 2]) continue;
            const int per_thread = pass % 2 == 0 ? 1 : 2;
            const int S = TW * TH, nblk = (g.K + kBlk - 1) / kBlk, SJ = TW + 2;
            if (nblk * S > per_thread * bt) continue;
            const int row = 9 * (g.K + 1) * SJ;
            int pad = 0;
            for (int x = 1; x < 32; x++)
                if (bank_conflicts(TW, S, SJ, row + x) < bank_conflicts(TW, S, SJ, row + pad))
                    pad = x;
            const int SYs = row + pad;
            const int words = (TH + 2) * SYs + kBlk * 9 * SJ;
            const int TN = S * g.K;
            const size_t bytes = (size_t)(words + nblk + 2 + TN + 1) * sizeof(int32_t);
            // (a list entry is a cell's 16-bit offset: 224 KB are 57344 words)
            if (bytes > 224 * 1024) continue;
            t.TW = TW;
            t.TH = TH;
            t.SJ = SJ;
            t.SYs = SYs;
            t.words = words;
            t.S = S;
            t.nblk = nblk;
            t.TN = TN;
            t.rTH = TH == 1 ? 0u : (unsigned)((0x100000000ull + TH - 1) / TH);
            t.rS = (unsigned)((0x100000000ull + S - 1) / S);
            t.tiles_w = (g.ng + TW - 1) / TW;
            t.tiles_h = (g.h + TH - 1) / TH;
            t.T = t.tiles_w * t.tiles_h;
            tpt = per_thread;
            smem = bytes;
            if (fields) *fields = fb;
            return true;
        }
    }
    return false;
}

// Threads per block for a pair: 256 when its options ask for it, but 512 for a
// shape that 8 nodes per thread of 256 hold and two blocks of whole layers do
// not (a number of layers that is not a multiple of kBlk).
static int cta_threads(const Geom &g, const gs_solve_opts *o) {
    if (o->cta_threads != 256) return 512;
    TileGeom t;
    int tpt;
    size_t smem;
    if (pick_tile(g, t, tpt, smem, o->tile_w, o->tile_h, 256)) return 256;
    const bool shape = o->tile_w == 4 || o->tile_w == 8 || o->tile_w == 16 || o->tile_w == 32;
    const size_t fb = shape && o->tile_h > 0 ? field_bytes(g, o->tile_w, o->tile_h, 256) : 0;
    return fb && fb <= 180 * 1024 ? 512 : 256;
}

// Per-tile flags are sized for the most tiles any allowed shape gives (4 x 1
// sites), so one workspace serves every tile shape.
static int64_t max_tiles(const Geom &g) { return (int64_t)((g.ng + 3) / 4) * g.h; }

size_t tiled_work_extra(const Geom &g) {
    return round_up(g.N * sizeof(uint16_t), 256) + round_up(8 * max_tiles(g) * sizeof(int32_t), 256);
}

// Per-pair arguments from the pair's geometry, state and workspace.
static int setup_args(const Geom &g, const State &s, const Work &w, const gs_solve_opts *o,
                      SolveArgs &a, int &tpt, size_t &smem, int bt) {
    memset(&a, 0, sizeof(a));
    a.g = g;
    a.s = s;
    if (!pick_tile(g, a.t, tpt, smem, o->tile_w, o->tile_h, bt)) return GS_ERR_INVAL;
    a.tpt = tpt;
    // a step's item count travels in 24 bits of the claim word
    if (a.t.T > (int)(kItemMask - 4096)) return GS_ERR_INVAL;
    char *extra = (char *)w.mark + round_up(g.N * sizeof(int32_t), 256);
    a.amask = (uint16_t *)extra;
    a.tile_act = (int32_t *)(extra + round_up(g.N * sizeof(uint16_t), 256));
    a.tile_dirty = a.tile_act + 2 * a.t.T;
    a.tile_cnt = a.tile_act + 4 * a.t.T;
    a.tile_list = a.tile_act + 5 * a.t.T;
    a.ctrl = w.ctrl;
    return GS_OK;
}

static void solve_fields(SolveArgs &a, const gs_solve_opts *o) {
    a.hgt = a.s.ht;
    a.dir = 0;
    a.mode = o->mode;
    a.sweeps_per_relabel = o->sweeps_per_relabel;
    a.local_iters = o->local_iters > 0 ? o->local_iters : 8;
    // a pass takes heights across one tile, so the cap grows as tiles shrink:
    // over eleven sizes 8 passes at 16 x 8 sites, 16 at 8 x 8 and 32 at 8 x 4
    // were the fastest of 8, 12, 16, 24 and 32 (271x144x62: 37.6 ms with 8, 27.5
    // with 32).  Tail visits of 2 x local_iters: 5 % less than 4 x (an iteration
    // is a whole block's now, not a warp's own).  In fixed-sweep mode the caller
    // counts rounds, and the time of an exact solve is no reason to do less in
    // one: 4 x there (384x288x16, 128 rounds: 0.0020 % of the flow still
    // missing, 0.0039 % with 2 x).
    a.relabel_passes = o->relabel_passes > 0 ? o->relabel_passes
                                             : std::min(64, std::max(8, 1024 / a.t.S));
    a.tail_iters = o->tail_iters > 0 ? o->tail_iters
                                     : (a.mode == GS_MODE_FIXED_SWEEPS ? 4 : 2) * a.local_iters;
    a.fixed_sweeps = o->fixed_sweeps;
    a.max_iters = o->max_iters;
}

// Cooperative launch of the batch kernel with the whole grid resident.  The
// launch goes through cudaLaunchKernelEx with the cooperative attribute, so a
// caller may capture it in a CUDA graph.
static int launch_batch(const BatchArgs &B, int tpt, size_t smem, int total_tiles, int bt,
                        cudaStream_t st) {
    void (*kern)(const BatchArgs) = tpt == 1 ? k_batch<1> : k_batch<2>;
    int dev = 0;
    GS_CUDA_TRY(cudaGetDevice(&dev));
    int sms = 0, coop = 0;
    GS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    GS_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return GS_ERR_CUDA;
    GS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    GS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, bt, smem));
    if (per_sm < 1) return GS_ERR_INVAL;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(per_sm * sms, total_tiles));
    cfg.blockDim = dim3(bt);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    GS_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, B));
    count_launches(1);
    return GS_OK;
}

// Control words of a batch launch: the abort flag and finished-pair count,
// then one PairCtl per pair.
constexpr size_t kBatchCtrlBytes = 256 + kMaxPairs * sizeof(PairCtl);
static_assert(512 + sizeof(PairCtl) <= kWorkCtrlBytes, "a pair's workspace holds its control words");

// Idle limit of a launch from one pair's options (0: the default); a batch
// takes the smallest.
static unsigned long long idle_limit_ns(const gs_solve_opts *o) {
    return o->idle_limit_us > 0 ? 1000ull * (unsigned long long)o->idle_limit_us
                                : kDefaultIdleLimitNs;
}

static int run_batch(BatchArgs &B, int tpt, size_t smem, int bt, void *ctrl_mem,
                     cudaStream_t st) {
    B.bar = (Ctrl *)ctrl_mem;
    B.ctl = (PairCtl *)((char *)ctrl_mem + 256);
    int total = 0;
    for (int p = 0; p < B.n; p++) total += B.pair[p].t.T;
    GS_CUDA_TRY(cudaMemsetAsync(ctrl_mem, 0, 256 + (size_t)B.n * sizeof(PairCtl), st));
    return launch_batch(B, tpt, smem, total, bt, st);
}

size_t batch_ctrl_bytes() { return kBatchCtrlBytes; }


int tiled_solve(const Geom &g, const State &s, const Work &w, const gs_solve_opts *o,
                int32_t *status, cudaStream_t st) {
    static BatchArgs B;   // host staging of the kernel argument (copied at launch)
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    memset(&B, 0, sizeof(B));
    B.n = 1;
    B.extract = 0;
    B.idle_limit_ns = idle_limit_ns(o);
    int tpt;
    size_t smem;
    const int bt = cta_threads(g, o);
    int rc = setup_args(g, s, w, o, B.pair[0], tpt, smem, bt);
    if (rc) return rc;
    solve_fields(B.pair[0], o);
    B.pair[0].status = status;
    GS_CUDA_TRY(cudaMemsetAsync(w.ctrl, 0, sizeof(Ctrl), st));
    return run_batch(B, tpt, smem, bt, (char *)w.ctrl + 256, st);
}

int tiled_extract(const Geom &g, const State &s, const Work &w, const gs_solve_opts *o,
                  int32_t *labels, int64_t *flow, int32_t *status, cudaStream_t st) {
    static BatchArgs B;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    memset(&B, 0, sizeof(B));
    B.n = 1;
    B.extract = 1;
    B.idle_limit_ns = idle_limit_ns(o);
    int tpt;
    size_t smem;
    const int bt = cta_threads(g, o);
    int rc = setup_args(g, s, w, o, B.pair[0], tpt, smem, bt);
    if (rc) return rc;
    SolveArgs &a = B.pair[0];
    a.hgt = w.mark;
    a.dir = o->mode == GS_MODE_EXACT ? 2 : 0;
    a.mode = GS_MODE_EXACT;
    a.max_iters = 1;
    a.labels = labels;
    a.flow = flow;
    a.status = status;
    return run_batch(B, tpt, smem, bt, (char *)w.ctrl + 256, st);
}

}  // namespace gs

extern "C" int gs_tile_info(const gs_params *p, const gs_solve_opts *o, int32_t *out) {
    gs::Geom g;
    if (gs::make_geom(p, &g) != GS_OK || !o || !out) return GS_ERR_INVAL;
    gs::TileGeom t;
    int tpt;
    size_t smem, fields;
    if (!gs::pick_tile(g, t, tpt, smem, o->tile_w, o->tile_h, gs::cta_threads(g, o), &fields))
        return GS_ERR_INVAL;
    out[0] = t.TW;
    out[1] = t.TH;
    out[2] = t.T;
    out[3] = (int32_t)fields;
    return GS_OK;
}

extern "C" size_t gs_tile_smem_bytes(const gs_params *p, const gs_solve_opts *o) {
    gs::Geom g;
    gs::TileGeom t;
    int tpt;
    size_t smem;
    if (!o || gs::make_geom(p, &g) != GS_OK ||
        !gs::pick_tile(g, t, tpt, smem, o->tile_w, o->tile_h, gs::cta_threads(g, o)))
        return 0;
    return smem;
}

// ------------------------------------------------------------ batched ABI ---

extern "C" size_t gs_batch_workspace_bytes(int32_t n) {
    if (n < 1 || n > gs::kMaxPairs) return 0;
    return gs::kBatchCtrlBytes;
}

extern "C" int gs_solve_batched(const gs_pair_desc *descs, int32_t n, void *batch_ws, void *stream) {
    using namespace gs;
    if (!descs || n < 1 || n > kMaxPairs || !batch_ws || ((uintptr_t)batch_ws & 255))
        return GS_ERR_INVAL;
    cudaStream_t st = (cudaStream_t)stream;
    static BatchArgs B, E;   // host staging of the kernel arguments (copied at launch)
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    memset(&B, 0, sizeof(B));
    memset(&E, 0, sizeof(E));
    B.n = E.n = n;
    B.extract = 0;
    E.extract = 1;
    B.idle_limit_ns = kDefaultIdleLimitNs;
    int tpt_max = 1;
    size_t smem_max = 0;
    // one block size for the launch: 256 threads only when every pair asks
    int bt = 256;
    for (int i = 0; i < n; i++) {
        Geom g;
        if (make_geom(&descs[i].p, &g) != GS_OK) return GS_ERR_INVAL;
        if (cta_threads(g, &descs[i].o) != 256) bt = 512;
    }
    for (int i = 0; i < n; i++) {
        const gs_pair_desc &d = descs[i];
        Geom g;
        if (make_geom(&d.p, &g) != GS_OK || !d.L || !d.R || !d.cost || !d.graph || !d.workspace ||
            !d.labels || !d.flow || !d.status)
            return GS_ERR_INVAL;
        if (gs_check_solve_opts(&d.o) != GS_OK || d.o.engine != GS_ENGINE_TILED ||
            ((uintptr_t)d.graph & 255) || ((uintptr_t)d.workspace & 255))
            return GS_ERR_INVAL;
        B.idle_limit_ns = std::min(B.idle_limit_ns, idle_limit_ns(&d.o));
        const State s = state_view(d.graph, g);
        const Work w = work_view(d.workspace, g);
        int tpt;
        size_t smem;
        if (setup_args(g, s, w, &d.o, B.pair[i], tpt, smem, bt) != GS_OK) return GS_ERR_INVAL;
        solve_fields(B.pair[i], &d.o);
        B.pair[i].status = d.status;
        E.pair[i] = B.pair[i];
        SolveArgs &x = E.pair[i];
        x.hgt = w.mark;
        x.dir = d.o.mode == GS_MODE_EXACT ? 2 : 0;
        x.mode = GS_MODE_EXACT;
        x.max_iters = 1;
        x.labels = d.labels;
        x.flow = d.flow;
        tpt_max = std::max(tpt_max, tpt);
        smem_max = std::max(smem_max, smem);
    }
    // per pair: data term and graph (small launches), then one launch for all
    // solves and one for all label extractions
    for (int i = 0; i < n; i++) {
        const gs_pair_desc &d = descs[i];
        int rc = gs_stereo_cost_volume(d.L, d.R, d.p.w, &d.p, d.cost, stream);
        if (rc) return rc;
        rc = gs_build_graph(d.cost, &d.p, d.graph, d.status, stream);
        if (rc) return rc;
        GS_CUDA_TRY(cudaMemsetAsync(B.pair[i].ctrl, 0, sizeof(Ctrl), st));
    }
    E.idle_limit_ns = B.idle_limit_ns;
    int rc = run_batch(B, tpt_max, smem_max, bt, batch_ws, st);
    if (rc) return rc;
    return run_batch(E, tpt_max, smem_max, bt, batch_ws, st);
}

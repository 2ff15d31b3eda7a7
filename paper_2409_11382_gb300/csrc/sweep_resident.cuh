// sweep_resident.cuh -- a multigrid cycle on the correction problem of a small
// level, all its levels resident in one thread-block cluster, in one launch.
//
// The small levels (up to a few thousand cells) are bound by latency, not by
// arithmetic or bytes: as one graph-launched kernel per sweep each costs a launch
// gap, a global round trip to stage a tile with its halo, and the barriers of a
// tile sweep.  Here a level's rows are dealt out to the CTAs of a cluster; a
// thread keeps its cell's state in registers over the sweeps of the level, and a
// sweep exchanges only m_s and the post-collision data through shared memory, the
// rows at the slab edges straight into the neighbour CTA's.  A sweep is two
// barriers: (B) the post-collision data of every row written, (A) m_s of every row
// updated.  Restriction and prolongation read the other level's rows through
// distributed shared memory.
//
// FP64 levels (the coarsest level of the FP32 path, every level of the FP64 path)
// are bound by FP64 instructions: one holds its SM sub-partition for 64 clocks
// whatever its number of active lanes (measured: latency 63, four warps on four
// sub-partitions one per 19).  Four lanes share a cell there, one per pair of
// opposite directions, so that a sweep issues 35 FP64 instructions per warp of 8
// cells (47 with a wall) where one lane per cell issued 124 (some 290 with the
// warp's wall cells) on mostly empty warps.
//
// The operations and their rounding are those of the strip and tile sweeps
// (collide_math, residual_core and the wall table), so results are bitwise those of
// separate launches.
#pragma once
#include "sweep_mom.cuh"

namespace biot {

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// The address of *p (this CTA's shared memory) in CTA `rank` of the cluster.
template <typename T>
__device__ __forceinline__ T *cluster_peer(T *p, int rank)
{
    T *q;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
    return q;
}

// Barrier of all threads of the cluster, ordering their shared-memory accesses.
__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// What the per-cell code reads of a level (fields of SweepArgs).
template <typename T>
struct ResView {
    int nx, ny;
    int bc[4];
    T *H[4];  // fullway bounce-back history, indexed by the cell's global position along the side
    T k_fs, k_hs, k_hd, k_h22, k_gam;
};
template <typename T>
struct WallKinds {  // the argument of wall_cell_index
    const int *bc;
    int nx, ny, hist_valid;
};

// Post-collision data of a level by (padded local row, column).
template <typename T>
struct SlabPost {
    const T *post;
    int nx, plane;
    __device__ __forceinline__ T at(int k, int s, int c) const { return post[k * plane + s * nx + c]; }
    __device__ __forceinline__ T G(int s, int k, int c) const { return at(k, s, c); }
    __device__ __forceinline__ T MX(int s, int c) const { return at(8, s, c); }
    __device__ __forceinline__ T MY(int s, int c) const { return at(9, s, c); }
};

// This CTA's part of one level: rows row0 .. row0 + rows - 1.
template <typename T>
struct Slab {
    T *m, *x;          // iterate (NM planes of cap), right-hand side (5 planes of cap)
    float *cvt;        // an FP64 level's iterate rounded to FP32, for an FP32 level above it
    T *ms, *post;      // m_s and post-collision planes of rpc + 2 rows (work areas shared by the levels)
    T *dres;           // residuals to be restricted, 5 planes of cap
    const unsigned *map;  // cells, interior ones first: x | local row << 16
    int nx, ny, rpc, nranks, cap, plane;
    int rank, row0, rows, ncell, nint;
    bool perx, pery;
    int down, up;          // ranks of the rows row0 - 1 and row0 + rows (-1: beyond a wall)
    int down_halo;         // padded row there that mirrors this slab's first row (its last row: row 0)
};

__device__ __forceinline__ int slab_rows(int ny, int rpc, int rank)
{
    const int left = ny - rank * rpc;
    return left < 0 ? 0 : left < rpc ? left : rpc;
}

template <typename T>
__device__ __forceinline__ Slab<T> make_slab(const ResProg &P, const ResLevel &L, unsigned char *smem, int rank)
{
    Slab<T> S;
    S.m = reinterpret_cast<T *>(smem + L.m);
    S.x = reinterpret_cast<T *>(smem + L.x);
    S.cvt = reinterpret_cast<float *>(smem + L.cvt);
    S.map = reinterpret_cast<const unsigned *>(smem + L.map);
    S.ms = reinterpret_cast<T *>(smem + P.ms);
    S.post = reinterpret_cast<T *>(smem + P.post);
    S.dres = reinterpret_cast<T *>(smem + P.dres);
    S.nx = L.nx;
    S.ny = L.ny;
    S.rpc = L.rpc;
    S.nranks = L.nranks;
    S.cap = L.rpc * L.nx;
    S.plane = (L.rpc + 2) * L.nx;
    S.rank = rank;
    S.row0 = rank * L.rpc;
    S.rows = slab_rows(L.ny, L.rpc, rank);
    S.ncell = S.rows * L.nx;
    S.perx = P.bc[SIDE_LEFT] == BC_PERIODIC;
    S.pery = P.bc[SIDE_BOTTOM] == BC_PERIODIC;
    const int ri = min(S.row0 + S.rows, L.ny - 1) - max(S.row0, 1);  // rows without row 0 and row ny - 1
    S.nint = (ri > 0 && L.nx > 2) ? ri * (L.nx - 2) : 0;
    const int yd = S.row0 - 1, yu = S.row0 + S.rows;
    S.down = yd >= 0 ? rank - 1 : S.pery ? L.nranks - 1 : -1;
    S.up = yu < L.ny ? rank + 1 : S.pery ? 0 : -1;
    S.down_halo = S.down >= 0 ? slab_rows(L.ny, L.rpc, S.down) + 1 : 0;
    return S;
}

// The slab's cells, interior cells first (so that whole warps run one form of the
// residual), then row 0, row ny - 1 and the two side columns.
__device__ __forceinline__ void slab_map(unsigned *map, int nx, int ny, int row0, int rows)
{
    const int r0 = max(row0, 1), r1 = min(row0 + rows, ny - 1), ri = max(r1 - r0, 0), ci = max(nx - 2, 0);
    const int nint = ri * ci, nlow = (row0 == 0 && rows > 0) ? nx : 0;
    const int nhigh = (ny > 1 && row0 < ny && row0 + rows == ny) ? nx : 0;
    const int n = rows * nx;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        int x, y;
        if (i < nint) {
            x = 1 + i % ci;
            y = r0 + i / ci;
        } else if (i < nint + nlow) {
            x = i - nint;
            y = 0;
        } else if (i < nint + nlow + nhigh) {
            x = i - nint - nlow;
            y = ny - 1;
        } else {
            const int k = i - nint - nlow - nhigh;
            x = k < ri ? 0 : nx - 1;
            y = r0 + (k < ri ? k : k - ri);
        }
        map[i] = (unsigned)x | (unsigned)(y - row0) << 16;
    }
}

// Where a cell's m_s and post-collision data also go: the halo rows of the
// neighbour slabs when it lies in its slab's first or last row (nullptr: nowhere).
// Beyond a wall the slab's own m_s halo row takes the adjacent cell (even
// extension of the divergence).
template <typename T>
struct Edge {
    T *ms_down = nullptr, *ms_up = nullptr, *post_down = nullptr, *post_up = nullptr;
};
template <typename T>
__device__ __forceinline__ Edge<T> slab_edge(const Slab<T> &S, int x, int ly)
{
    Edge<T> e;
    if (ly == 0) {
        e.ms_down = S.ms + x;
        if (S.down >= 0) {
            e.ms_down = cluster_peer(S.ms, S.down) + S.down_halo * S.nx + x;
            e.post_down = cluster_peer(S.post, S.down) + S.down_halo * S.nx + x;
        }
    }
    if (ly == S.rows - 1) {
        e.ms_up = S.ms + (S.rows + 1) * S.nx + x;
        if (S.up >= 0) {
            e.ms_up = cluster_peer(S.ms, S.up) + x;
            e.post_up = cluster_peer(S.post, S.up) + x;
        }
    }
    return e;
}
template <typename T>
__device__ __forceinline__ void put_ms(const Slab<T> &S, const Edge<T> &e, int x, int ly, T v)
{
    S.ms[(ly + 1) * S.nx + x] = v;
    if (e.ms_down) *e.ms_down = v;
    if (e.ms_up) *e.ms_up = v;
}

// Barrier of the threads that hold the level: `live` threads of this CTA when it
// holds the whole level, else the cluster (the CTAs without rows keep step).
__device__ __forceinline__ void level_barrier(int nranks, int rank, int live)
{
    if (nranks > 1) cluster_barrier();
    else if (rank == 0 && (int)threadIdx.x < live) asm volatile("bar.sync 1, %0;" ::"r"(live) : "memory");
}

// A cell on four lanes: lane p of the quad holds pair p of the directions, and of
// the cell's state m_10 | m_01 | m_11 | m_s by lane, m_d on every lane (and m_12 |
// m_21 | m_22 on lanes 0 to 2).  Operands are selected per lane so that one
// instruction serves the quad; each value is formed by the operations of
// collide_math and residual_core, in their order.
template <typename T, int KIND>
struct QuadCell {
    static_assert(!kind_fine(KIND), "correction problems");
    static constexpr bool GH = kind_ghosts(KIND);
    static constexpr unsigned FULL = 0xffffffffu, SIGN = 0x80000000u;
    int id, p, x, ly, i, y;
    bool mine, axis, walls, border;
    int g_hi, g_lo, g_c1, g_c2, g_ne, g_sw;  // lanes 0 / 1: cells of the x / y gradient in the padded m_s
    int k0, k1;                              // the pair's directions (pair_first, pair_second)
    Edge<T> edge;
    T mp, m4, rp, r4, mg;    // state and right-hand side
    T v, tx, ty, gp, gm;     // collision input (component p; 10; 01), outgoing populations
    // the wall table's entry: descriptors of the two pulls with their source
    // offsets, beta coefficients of component p, of m_d and of the ghost moment
    unsigned d0, d1;
    int o0, o1, q0, q1;
    T cp[2], c4[2], cg[2];
    bool beta;

    __device__ __forceinline__ T from(T a, int lane) const { return __shfl_sync(FULL, a, lane, 4); }

    // lane t of the quads of the cells first, first + 1, ... of the slab's list
    __device__ __forceinline__ void init(const Slab<T> &S, int t, int first)
    {
        id = first + (t >> 2);
        p = t & 3;
        mine = t >= 0 && id < S.ncell;
        border = mine && id >= S.nint;
        axis = p < 2;
        const unsigned xy = mine ? S.map[id] : 0;
        x = xy & 0xffff;
        ly = xy >> 16;
        i = ly * S.nx + x;
        y = S.row0 + ly;
        const int xm = x > 0 ? x - 1 : S.perx ? S.nx - 1 : 0, xp = x < S.nx - 1 ? x + 1 : S.perx ? 0 : S.nx - 1;
        const int ib = ly * S.nx, io = ib + S.nx, ia = io + S.nx;  // rows below, own, above of the padded m_s
        g_hi = p == 1 ? ia + x : io + xp;
        g_lo = p == 1 ? ib + x : io + xm;
        g_c1 = p == 1 ? ia + xm : ib + xp;  // NE + c1, c2 + SW
        g_c2 = p == 1 ? ib + xp : ia + xm;
        g_ne = ia + xp;
        g_sw = ib + xm;
        k0 = p == 0 ? 0 : p == 1 ? 1 : p == 2 ? 4 : 5;
        k1 = p == 0 ? 2 : p == 1 ? 3 : p == 2 ? 6 : 7;
        mp = m4 = rp = r4 = mg = T(0);
        if (mine) {
            edge = slab_edge(S, x, ly);
            mp = S.m[p * S.cap + i];
            m4 = S.m[4 * S.cap + i];
            rp = S.x[p * S.cap + i];
            r4 = S.x[4 * S.cap + i];
            if (GH && p < 3) mg = S.m[(5 + p) * S.cap + i];
        }
        walls = __any_sync(FULL, border);
    }
    __device__ __forceinline__ void pull_offset(const Slab<T> &S, unsigned d, int &o, int &q) const
    {
        int c = x - 1 + (int)((d >> WP_COL) & 3);
        c = c < 0 ? c + S.nx : c >= S.nx ? c - S.nx : c;  // a periodic level wraps
        o = (ly + (int)((d >> WP_ROW) & 3)) * S.nx + c;
        q = (int)(d & WP_K) * S.plane + o;
    }
    __device__ __forceinline__ void entry(const ResView<T> &a, const Slab<T> &S, int hist)
    {
        const WallKinds<T> k{a.bc, a.nx, a.ny, hist};
        const int wi = border ? wall_cell_index(k, x, y, S.perx, S.pery) : 0;
        const WallEntry<T> &E = wall_table<T>().e[wi];
        d0 = E.pull[k0];
        d1 = E.pull[k1];
        pull_offset(S, d0, o0, q0);
        pull_offset(S, d1, o1, q1);
        beta = false;
        if (walls) {
            beta = __any_sync(FULL, E.beta != 0);
#pragma unroll
            for (int c = 0; c < 2; c++) {
                cp[c] = p < 2 ? E.bd[p & 1][c] : E.bs[p & 1][c];
                c4[c] = E.bs[2][c];
                if constexpr (GH) cg[c] = wall_table<T>().g[wi].b[p < 3 ? p : 0][c];
            }
        }
    }
    __device__ __forceinline__ void collide(const ResView<T> &a, const Slab<T> &S)
    {
        v = mp - rp;  // collision input (lane p: component p; m_d everywhere)
        const T w = m4 - r4;
        const T *D = S.ms;
        const T f1 = D[g_hi] - D[g_lo];
        const T f2 = (D[g_ne] + D[g_c1]) - (D[g_c2] + D[g_sw]);
        const T F = mul_rn(a.k_fs, mad_rn(f1, T(1.0 / 3.0), mul_rn(f2, T(1.0 / 12.0))));
        const T Fx = from(F, 0), Fy = from(F, 1), c3 = from(v, 3), c2 = from(v, 2);
        tx = from(v, 0);
        ty = from(v, 1);
        const T Fd = Fy + flip_sign(Fx, p == 3 ? SIGN : 0u);
        const T Fs = p == 0 ? Fx : p == 1 ? Fy : Fd;
        const T t = mul_rn(axis ? a.k_hd : a.k_h22, axis ? w : c3);
        const T ks = flip_sign(axis ? a.k_hs : a.k_hd, p == 3 ? SIGN : 0u);
        const T hS = mad_rn(ks, axis ? c3 : c2, flip_sign(t, p == 1 ? SIGN : 0u));
        const T cb = axis ? T(5.0 / 12.0) : T(1.0 / 24.0);
        gp = mad_rn(cb, Fs, hS);
        gm = mad_rn(flip_sign(cb, SIGN), Fs, hS);
        if (!mine) return;
        const int pl = S.plane;
        T *q = S.post + (ly + 1) * S.nx + x;
        q[k0 * pl] = gp;
        q[k1 * pl] = gm;
        if (axis) q[(8 + p) * pl] = v;
        if (edge.post_down) {  // downward directions: the second of pairs 1 to 3, and the moments
            if (p > 0) edge.post_down[k1 * pl] = gm;
            if (axis) edge.post_down[(8 + p) * pl] = v;
        }
        if (edge.post_up) {
            if (p > 0) edge.post_up[k0 * pl] = gp;
            if (axis) edge.post_up[(8 + p) * pl] = v;
        }
    }
    __device__ __forceinline__ void pull(const ResView<T> &a, const Slab<T> &S, unsigned d, int o, int q, int k, int ko, T &g,
                                         T &h) const
    {
        const int pl = S.plane;
        g = flip_sign(S.post[q], d << (31 - WP_SG));
        const T dx = S.post[8 * pl + o] - tx, dy = S.post[9 * pl + o] - ty;
        const T dd = dy + flip_sign(dx, d << (31 - WP_SD));
        h = flip_sign(mul_rn(axis ? T(1.0 / 3.0) : T(1.0 / 12.0), p == 0 ? dx : p == 1 ? dy : dd), d << (31 - WP_SH));
        if (d & WP_HIST) {  // eq. BC:elasticity: the outgoing population of the previous call
            const int side = (d & WP_HOR) ? (ey8(k) > 0 ? SIDE_BOTTOM : SIDE_TOP) : (ex8(k) > 0 ? SIDE_LEFT : SIDE_RIGHT);
            g = a.H[side][3 * ((d & WP_HOR) ? x : y) + hslot(side, ko)];
            h = T(0);
        }
    }
    __device__ __forceinline__ void residual(const ResView<T> &a, const Slab<T> &S, bool restriction)
    {
        T g0, h0, g1, h1;
        pull(a, S, d0, o0, q0, k0, k1, g0, h0);
        pull(a, S, d1, o1, q1, k1, k0, g1, h1);
        const T Ss = (g0 + g1) + (h0 + h1), As = (g0 - g1) + (h0 - h1);
        const T A2 = from(As, 2), A3 = from(As, 3);
        const T S0 = from(Ss, 0), S1 = from(Ss, 1), S2 = from(Ss, 2), S3 = from(Ss, 3);
        //            lane 0: A0 + A2   1: A1 + A2   2: S2 - S3   3: S0 + S1
        const T t1 = (axis ? As : p == 2 ? S2 : S0) + flip_sign(axis ? A2 : p == 2 ? S3 : S1, p == 2 ? SIGN : 0u);
        //            lane 0: t1 - A3   1: t1 + A3   2: S0 - S1   3: S2 + S3
        const T t2 = (axis ? t1 : p == 2 ? S0 : S2) + flip_sign(axis ? A3 : p == 2 ? S1 : S3, (p & 1) ? 0u : SIGN);
        const T rr = mp - v;  // r_0 | r_1 as the residual forms them
        //            lane 0: r0 - t2   1: r1 - t2   2: m_11 - t1   3: t1 + 2 t2
        T d = mad_rn(p == 3 ? T(2) : T(-1), p == 2 ? t1 : t2, axis ? rr : p == 2 ? mp : t1);
        //            lane 2: d_4 = m_d - (S0 - S1)   3: d_3 = m_s - d
        const T d34 = (p == 3 ? mp : m4) - (p == 3 ? d : t2);
        if (p == 3) d = d34;
        T d4 = from(d34, 2), dg = T(0);
        if constexpr (GH) {  // ghost moments: d_5 | d_6 | d_7 on lanes 0 to 2
            const T u = (p == 2 ? S2 : A2) + flip_sign(axis ? A3 : S3, p == 0 ? SIGN : 0u);
            const T b = mul_rn(p == 0 ? tx : ty, T(1.0 / 3.0));
            dg = (p < 2 ? mg - b : mg) - u;
        }
        if (beta) {
            d -= mul_rn(cp[0], tx) + mul_rn(cp[1], ty);
            d4 -= mul_rn(c4[0], tx) + mul_rn(c4[1], ty);
            if constexpr (GH) dg -= mul_rn(cg[0], tx) + mul_rn(cg[1], ty);
        }
        if (border) {  // history of the fullway bounce-back: this call's outgoing populations
            const bool hb = y == 0 && a.bc[SIDE_BOTTOM] == BC_DIRICHLET, ht = y == a.ny - 1 && a.bc[SIDE_TOP] == BC_DIRICHLET;
            const bool hl = x == 0 && a.bc[SIDE_LEFT] == BC_DIRICHLET, hr = x == S.nx - 1 && a.bc[SIDE_RIGHT] == BC_DIRICHLET;
            if (hb || ht || hl || hr) {
                // beta of the pair's first direction (the second's is its negative)
                const T bx = p == 0 ? T(0.5 * pa_x(0)) : p == 1 ? T(0) : p == 2 ? T(0.5 * pa_x(2)) : T(0.5 * pa_x(3));
                const T by = p == 0 ? T(0) : p == 1 ? T(0.5 * pa_y(1)) : T(0.5 * pa_y(2));
                const T bm = mul_rn(bx, tx) + mul_rn(by, ty);
                const T out0 = gp + bm, out1 = gm - bm;
                if (hb && p > 0) a.H[SIDE_BOTTOM][3 * x + hslot(SIDE_BOTTOM, k1)] = out1;
                if (ht && p > 0) a.H[SIDE_TOP][3 * x + hslot(SIDE_TOP, k0)] = out0;
                if (hl && p != 1) a.H[SIDE_LEFT][3 * y + hslot(SIDE_LEFT, p == 3 ? k0 : k1)] = p == 3 ? out0 : out1;
                if (hr && p != 1) a.H[SIDE_RIGHT][3 * y + hslot(SIDE_RIGHT, p == 3 ? k1 : k0)] = p == 3 ? out1 : out0;
            }
        }
        if (restriction) {
            if (mine) {
                S.dres[p * S.cap + i] = d;
                if (p == 0) S.dres[4 * S.cap + i] = d4;
            }
        } else {
            const T ngam = flip_sign(a.k_gam, SIGN);
            mp = mad_rn(ngam, d, mp);
            m4 = mad_rn(ngam, d4, m4);
            if constexpr (GH) mg = mad_rn(ngam, dg, mg);
            if (mine && p == 3) put_ms(S, edge, x, ly, mp);
        }
    }
    __device__ __forceinline__ void store(const Slab<T> &S, bool to_fp32) const
    {
        if (!mine) return;
        S.m[p * S.cap + i] = mp;
        if (p == 0) S.m[4 * S.cap + i] = m4;
        if (GH && p < 3) S.m[(5 + p) * S.cap + i] = mg;
        if (to_fp32) {
            S.cvt[p * S.cap + i] = (float)mp;
            const float f4 = (float)m4;
            if (p == 0) S.cvt[4 * S.cap + i] = f4;
            if (GH) {
                const float fg = (float)mg;
                if (p < 3) S.cvt[(5 + p) * S.cap + i] = fg;
            }
        }
    }
};

// A cell away from the walls on one thread (FP32 levels).
template <int KIND>
struct InnerCell {
    using T = float;
    using L = RingLayout<KIND, false>;
    static constexpr int NM = kind_ghosts(KIND) ? 8 : 5;
    int x, ly, i;
    bool mine;
    Edge<T> edge;
    T m[8], e[L::NE];
    __device__ __forceinline__ void init(const Slab<T> &S, int id)
    {
        mine = id < S.nint;
        const unsigned xy = mine ? S.map[id] : 0x10000u;
        x = xy & 0xffff;
        ly = xy >> 16;
        i = ly * S.nx + x;
        if (!mine) return;
        edge = slab_edge(S, x, ly);
#pragma unroll
        for (int k = 0; k < NM; k++) m[k] = S.m[k * S.cap + i];
#pragma unroll
        for (int k = 0; k < L::NXV; k++) e[L::EX + k] = S.x[k * S.cap + i];
    }
    __device__ __forceinline__ void collide(const ResView<T> &a, const Slab<T> &S) const
    {
        if (!mine) return;
        const int nx = S.nx, pl = S.plane;
        const T *r0 = S.ms + ly * nx + x, *r1 = r0 + nx, *r2 = r1 + nx;
        const CollideOut<T> o = collide_math<T, KIND, false, L::NE>(a, m[0], m[1], m[2], m[3], m[4], e, r1[1], r1[-1], r2[0],
                                                                    r0[0], r2[1], r2[-1], r0[1], r0[-1]);
        T *q = S.post + (ly + 1) * nx + x;
#pragma unroll
        for (int k = 0; k < 8; k++) q[k * pl] = o.G[k];
        q[8 * pl] = o.mx;
        q[9 * pl] = o.my;
        if (edge.post_down) {  // the row below pulls the downward directions
            T *d = edge.post_down;
            d[3 * pl] = o.G[3];
            d[6 * pl] = o.G[6];
            d[7 * pl] = o.G[7];
            d[8 * pl] = o.mx;
            d[9 * pl] = o.my;
        }
        if (edge.post_up) {  // the row above the upward ones
            T *u = edge.post_up;
            u[1 * pl] = o.G[1];
            u[4 * pl] = o.G[4];
            u[5 * pl] = o.G[5];
            u[8 * pl] = o.mx;
            u[9 * pl] = o.my;
        }
    }
    __device__ __forceinline__ void residual(const ResView<T> &a, const Slab<T> &S, bool restriction)
    {
        if (!mine) return;
        if constexpr (kind_ghosts(KIND)) {
            e[0] = m[5];
            e[1] = m[6];
            e[2] = m[7];
        }
        const OwnCell<T> own = own_from<T, KIND, false, L::NE>(m[0], m[1], m[2], m[3], m[4], e);
        const int sl[3] = {ly, ly + 1, ly + 2};
        const WallTable<T> &W = wall_table<T>();
        T d[8];
        residual_cell<T, KIND, false, false>(a, SlabPost<T>{S.post, S.nx, S.plane}, x, 0, sl, x, own, d, W.e[0], W.g[0]);
        if (restriction) {
#pragma unroll
            for (int k = 0; k < 5; k++) S.dres[k * S.cap + i] = d[k];
        } else {
            const T gam = a.k_gam;
#pragma unroll
            for (int k = 0; k < NM; k++) m[k] = mad_rn(-gam, d[k], m[k]);
            put_ms(S, edge, x, ly, m[3]);
        }
    }
    __device__ __forceinline__ void store(const Slab<T> &S) const
    {
        if (!mine) return;
#pragma unroll
        for (int k = 0; k < NM; k++) S.m[k * S.cap + i] = m[k];
    }
};

// n smoothing sweeps of a level, or the residuals of its iterate into dres.
// FP64: every cell on four lanes; FP32: the cells away from the walls on one
// thread each (whole warps), the wall cells on four lanes each behind them.
// hist: the bounce-back history is valid.
template <typename T, int KIND>
__device__ __forceinline__ void level_sweeps(const ResView<T> &a, const Slab<T> &S, int n, bool restriction, int hist, bool to_fp32)
{
    constexpr bool F32 = sizeof(T) == 4;
    const int base = F32 ? (S.nint + 31) & ~31 : 0, first = F32 ? S.nint : 0;
    const int live = base + ((4 * (S.ncell - first) + 31) & ~31);
    const int t = threadIdx.x;
    if (t >= live) {  // warps without cells only keep step
        for (int s = 0; s < n; s++) {
            level_barrier(S.nranks, S.rank, live);
            if (!restriction) level_barrier(S.nranks, S.rank, live);
        }
    } else if (F32 && t < base) {
        if constexpr (F32) {
            InnerCell<KIND> c;
            c.init(S, t);
            for (int s = 0; s < n; s++) {
                c.collide(a, S);
                level_barrier(S.nranks, S.rank, live);  // (B)
                c.residual(a, S, restriction);
                if (!restriction) level_barrier(S.nranks, S.rank, live);  // (A)
            }
            if (!restriction) c.store(S);
        }
    } else {
        QuadCell<T, KIND> c;
        c.init(S, t - base, first);
        c.entry(a, S, hist);
        for (int s = 0; s < n; s++) {
            c.collide(a, S);
            level_barrier(S.nranks, S.rank, live);  // (B)
            c.residual(a, S, restriction);
            if (!hist) {  // the walls' later sweeps read the history
                hist = 1;
                c.entry(a, S, 1);
            }
            if (!restriction) level_barrier(S.nranks, S.rank, live);  // (A)
        }
        if (!restriction) c.store(S, to_fp32);
    }
}

// The right-hand side of the next coarser level C from the residuals of level F
// (full-sum restriction, eq. MG:restriction: rows first, then columns), and its
// zero iterate.  One thread per (cell, moment): FP64 conversions and sums are few
// per warp.
template <typename T, typename TC, bool GH>
__device__ __forceinline__ void slab_restrict(const ResLevel &LF, const Slab<T> &F, const Slab<TC> &C)
{
    constexpr int NM = GH ? 8 : 5;
    if (C.rank >= C.nranks) return;
    const int n = (C.ncell + 31) & ~31;  // a moment's cells start at a warp
    for (int t = threadIdx.x; t < NM * n; t += blockDim.x) {
        const int k = t / n, id = t - k * n;
        if (id >= C.ncell) continue;
        const unsigned xy = C.map[id];
        const int x = xy & 0xffff, ly = xy >> 16, i = ly * C.nx + x, yf = 2 * (C.row0 + ly);
        C.m[k * C.cap + i] = TC(0);
        if (k >= 5) continue;
        const int ra = (int)((unsigned)yf * LF.inv >> 20), rb = (int)((unsigned)(yf + 1) * LF.inv >> 20);  // yf / F.rpc
        const T *pa = cluster_peer(F.dres, ra) + k * F.cap + (yf - ra * F.rpc) * F.nx + 2 * x;
        const T *pb = cluster_peer(F.dres, rb) + k * F.cap + (yf + 1 - rb * F.rpc) * F.nx + 2 * x;
        const T a0 = pa[0], a1 = pa[1], b0 = pb[0], b1 = pb[1];
        const TC r0 = (TC)(a0 + b0), r1 = (TC)(a1 + b1);
        C.x[k * C.cap + i] = r0 + r1;
    }
    for (int i = threadIdx.x; i < (C.rows + 2) * C.nx; i += blockDim.x) C.ms[i] = TC(0);
}

// The coarse correction of level C added to the iterate of level F.
template <typename T, typename TC, bool GH>
__device__ __forceinline__ void slab_prolong(const Slab<T> &F, const ResLevel &LC, const Slab<TC> &C)
{
    constexpr int NM = GH ? 8 : 5;
    if (F.rank >= F.nranks) return;
    for (int id = threadIdx.x; id < F.ncell; id += blockDim.x) {
        const unsigned xy = F.map[id];
        const int x = xy & 0xffff, ly = xy >> 16, i = ly * F.nx + x, yc = (F.row0 + ly) >> 1;
        const int rc = (int)((unsigned)yc * LC.inv >> 20), o = (yc - rc * C.rpc) * C.nx + (x >> 1);  // yc / C.rpc
        const Edge<T> edge = slab_edge(F, x, ly);
        T c[NM];
        if constexpr (sizeof(T) == 4 && sizeof(TC) == 8) {
            const float *q = cluster_peer(C.cvt, rc) + o;
#pragma unroll
            for (int k = 0; k < NM; k++) c[k] = q[k * C.cap];
        } else {
            const TC *q = cluster_peer(C.m, rc) + o;
#pragma unroll
            for (int k = 0; k < NM; k++) c[k] = q[k * C.cap];
        }
#pragma unroll
        for (int k = 0; k < NM; k++) {
            const T v = F.m[k * F.cap + i] + c[k];
            F.m[k * F.cap + i] = v;
            if (k == 3) put_ms(F, edge, x, ly, v);
        }
    }
}

// The level views, one per level of the program (only the member of the level's
// storage type is used).
struct ResViews {
    ResView<float> f[RES_MAX_LEVELS];
    ResView<double> d[RES_MAX_LEVELS];
    int hist[RES_MAX_LEVELS];
};

template <typename T>
__device__ __forceinline__ void res_view(ResView<T> &v, const ResProg &P, const ResLevel &L, unsigned char *smem, int rank,
                                         const T (&k)[5])
{
    v.nx = L.nx;
    v.ny = L.ny;
    T *H = reinterpret_cast<T *>(smem + L.H);  // bottom, top: 3 nx; left, right: 3 rpc
    const int shift = 3 * rank * L.rpc;        // left / right records are indexed by the global row
    v.H[SIDE_BOTTOM] = H;
    v.H[SIDE_TOP] = H + 3 * L.nx;
    v.H[SIDE_LEFT] = H + 6 * L.nx - shift;
    v.H[SIDE_RIGHT] = H + 6 * L.nx + 3 * L.rpc - shift;
    for (int s = 0; s < 4; s++) v.bc[s] = P.bc[s];
    v.k_fs = k[0];
    v.k_hs = k[1];
    v.k_hd = k[2];
    v.k_h22 = k[3];
    v.k_gam = k[4];
}

// The K smoothing sweeps, or one residual evaluation, of level l of the program.
template <bool GH>
__device__ __forceinline__ void res_level(const ResProg &P, const ResViews &V, unsigned char *smem, int rank, int l, int n,
                                          bool restriction, int hist)
{
    constexpr int KIND = KIND_COARSE | (GH ? 0 : KIND_NOGHOST);
    const ResLevel &L = P.lev[l];
    if (L.fp64) {
        level_sweeps<double, KIND>(V.d[l], make_slab<double>(P, L, smem, rank), n, restriction, hist,
                                   l > 0 && !P.lev[l - 1].fp64);
    } else {
        level_sweeps<float, KIND>(V.f[l], make_slab<float>(P, L, smem, rank), n, restriction, hist, false);
    }
}

// Barrier around a transfer between levels l and l + 1: of the CTAs that hold one
// of them.
__device__ __forceinline__ void transfer_barrier(const ResProg &P, int l, int rank)
{
    if (P.lev[l].nranks > 1 || P.lev[l + 1].nranks > 1) cluster_barrier();
    else if (rank == 0) __syncthreads();
}

// Storage-type dispatch of a transfer between levels l and l + 1.
template <bool GH>
__device__ __forceinline__ void res_transfer(const ResProg &P, unsigned char *smem, int rank, int l, bool down)
{
    const ResLevel &F = P.lev[l], &C = P.lev[l + 1];
    if (F.fp64) {
        const Slab<double> f = make_slab<double>(P, F, smem, rank), c = make_slab<double>(P, C, smem, rank);
        if (down) slab_restrict<double, double, GH>(F, f, c);
        else slab_prolong<double, double, GH>(f, C, c);
    } else if (C.fp64) {
        const Slab<float> f = make_slab<float>(P, F, smem, rank);
        const Slab<double> c = make_slab<double>(P, C, smem, rank);
        if (down) slab_restrict<float, double, GH>(F, f, c);
        else slab_prolong<float, double, GH>(f, C, c);
    } else {
        const Slab<float> f = make_slab<float>(P, F, smem, rank), c = make_slab<float>(P, C, smem, rank);
        if (down) slab_restrict<float, float, GH>(F, f, c);
        else slab_prolong<float, float, GH>(f, C, c);
    }
}

// The bounce-back history of the top level between its slab and global memory
// (the records of the cells this CTA holds).
template <typename T>
__device__ __forceinline__ void res_history(const ResProg &P, const ResView<T> &v, const Slab<T> &S, bool load)
{
    for (int s = 0; s < 4; s++) {
        if (P.bc[s] != BC_DIRICHLET) continue;
        const bool horiz = s == SIDE_BOTTOM || s == SIDE_TOP;
        if (s == SIDE_BOTTOM && S.row0 != 0) continue;
        if (s == SIDE_TOP && S.row0 + S.rows != S.ny) continue;
        T *g = static_cast<T *>(P.H[s]);
        const int i0 = horiz ? 0 : 3 * S.row0, n = horiz ? 3 * S.nx : 3 * S.rows;
        for (int i = i0 + threadIdx.x; i < i0 + n; i += blockDim.x) {
            if (load) v.H[s][i] = g[i];
            else g[i] = v.H[s][i];
        }
    }
}

// The correction problem of the top level: its right-hand side, and its iterate
// (zero, or the stored one with its history).
template <typename T, bool GH>
__device__ __forceinline__ void res_load(const ResProg &P, const ResView<T> &v, unsigned char *smem, int rank)
{
    constexpr int NM = GH ? 8 : 5;
    const Slab<T> S = make_slab<T>(P, P.lev[0], smem, rank);
    if (!S.ncell) return;
    const size_t NP = (size_t)S.nx * S.ny;
    const T *r = static_cast<const T *>(P.r) + (size_t)S.row0 * S.nx;
    const T *g = static_cast<const T *>(P.g) + (size_t)S.row0 * S.nx;
    for (int i = threadIdx.x; i < S.ncell; i += blockDim.x) {
#pragma unroll
        for (int k = 0; k < 5; k++) S.x[k * S.cap + i] = r[k * NP + i];
#pragma unroll
        for (int k = 0; k < NM; k++) S.m[k * S.cap + i] = P.zero ? T(0) : g[k * NP + i];
    }
    // m_s with its halo rows: the rows beyond the slab's edges come from the stored iterate too
    for (int i = threadIdx.x; i < (S.rows + 2) * S.nx; i += blockDim.x) {
        T ms = T(0);
        if (!P.zero) {
            const int ly = i / S.nx, x = i - ly * S.nx;
            int y = S.row0 + ly - 1;
            y = S.pery ? wrapi(y, S.ny) : clampi(y, S.ny);
            ms = static_cast<const T *>(P.g)[3 * NP + (size_t)y * S.nx + x];
        }
        S.ms[i] = ms;
    }
    if (P.hist_valid) res_history<T>(P, v, S, true);
}

template <typename T, bool GH>
__device__ __forceinline__ void res_store(const ResProg &P, const ResView<T> &v, unsigned char *smem, int rank)
{
    constexpr int NM = GH ? 8 : 5;
    const Slab<T> S = make_slab<T>(P, P.lev[0], smem, rank);
    if (!S.ncell) return;
    T *g = static_cast<T *>(P.g) + (size_t)S.row0 * S.nx;
    const size_t NP = (size_t)S.nx * S.ny;
    for (int i = threadIdx.x; i < S.ncell; i += blockDim.x) {
#pragma unroll
        for (int k = 0; k < NM; k++) g[k * NP + i] = S.m[k * S.cap + i];
    }
    if (P.keep_hist) res_history<T>(P, v, S, false);
}

// Cluster blockIdx.x / cs runs program blockIdx.x / cs: one cycle on the
// correction problem of the program's top level.
template <bool GH>
__global__ void __launch_bounds__(RES_NT) k_resident_cycle(const __grid_constant__ ResParams PP)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ResViews V;
    __shared__ ResProg P;  // the program, out of the parameter block (constant-cache misses on every level change)
    {
        const int *src = reinterpret_cast<const int *>(&PP.p[blockIdx.x / PP.cs]);
        for (int i = threadIdx.x; i < (int)(sizeof(ResProg) / sizeof(int)); i += RES_NT) reinterpret_cast<int *>(&P)[i] = src[i];
    }
    __syncthreads();
    const int rank = (int)cluster_rank();
    if (threadIdx.x < P.nlev) {
        const int l = threadIdx.x;
        if (P.lev[l].fp64) res_view<double>(V.d[l], P, P.lev[l], smem, rank, P.kd);
        else res_view<float>(V.f[l], P, P.lev[l], smem, rank, P.kf);
        V.hist[l] = l == 0 ? P.hist_valid : 0;
    }
    for (int l = 0; l < P.nlev; l++) {
        const ResLevel &L = P.lev[l];
        slab_map(reinterpret_cast<unsigned *>(smem + L.map), L.nx, L.ny, rank * L.rpc, slab_rows(L.ny, L.rpc, rank));
    }
    __syncthreads();
    if (P.lev[0].fp64) res_load<double, GH>(P, V.d[0], smem, rank);
    else res_load<float, GH>(P, V.f[0], smem, rank);
    cluster_barrier();  // every CTA's rows set up (and every CTA of the cluster running)
    for (int i = 0; i < P.nops; i++) {
        const int l = P.ops[i] & RES_OP_LEVEL, op = P.ops[i] & ~RES_OP_LEVEL;
        if (op == RES_OP_SMOOTH) {
            int n = P.lev[l].K;
            while (i + 1 < P.nops && P.ops[i + 1] == P.ops[i]) {  // the coarsest level's two runs in one
                n += P.lev[l].K;
                i++;
            }
            const int hist = V.hist[l];
            res_level<GH>(P, V, smem, rank, l, n, false, hist);
            __syncthreads();
            if (threadIdx.x == 0) V.hist[l] = 1;  // read after a later barrier
        } else if (op == RES_OP_DOWN) {
            res_level<GH>(P, V, smem, rank, l, 1, true, 1);
            transfer_barrier(P, l, rank);  // residuals of every row written, the work areas free
            res_transfer<GH>(P, smem, rank, l, true);
            if (threadIdx.x == 0) V.hist[l + 1] = 0;
            transfer_barrier(P, l, rank);
        } else {
            transfer_barrier(P, l, rank);  // level l + 1 finished, the work areas free
            res_transfer<GH>(P, smem, rank, l, false);
            transfer_barrier(P, l, rank);
        }
    }
    __syncthreads();
    if (P.lev[0].fp64) res_store<double, GH>(P, V.d[0], smem, rank);
    else res_store<float, GH>(P, V.f[0], smem, rank);
    cluster_barrier();  // no CTA leaves while another may still write into its shared memory
}

template <bool GH>
cudaError_t resident_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at, int clusters, int cs, size_t smem, cudaStream_t s)
{
    auto kern = k_resident_cycle<GH>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM_MAX);
    if (e == cudaSuccess && cs > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cfg = {};
    cfg.gridDim = dim3(clusters * cs, 1, 1);
    cfg.blockDim = dim3(RES_NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cs;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return e;
}

template <bool GH>
cudaError_t launch_resident_kind(const ResParams &P, size_t smem, cudaStream_t s)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    cudaError_t e = resident_config<GH>(cfg, at[0], P.nprog, P.cs, smem, s);
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, k_resident_cycle<GH>, P) : e;
}

}  // namespace biot

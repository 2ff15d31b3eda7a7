// wall_table.cuh -- how the eight pulls of a wall cell find their populations, as
// a table indexed by the walls the cell touches.
//
// Whatever the wall, a pull across it takes direction K with its x and/or y
// component reversed, read in the cell's own column and/or row (a mirror reverses
// the component normal to the wall, a bounce-back both, §3.6); what differs are
// signs, and the beta terms of the residual (sweep_mom.cuh).  All of that is fixed
// by the walls at the cell, so it is evaluated at compile time, in the order of
// operations of the residual: the wall form of a sweep then loads one entry and
// runs the same straight code for every kind of wall.  As nested branches the
// pulls of a warp of border cells ran up to 40 divergent pieces one after the
// other, and their beta terms cost some 100 more operations per cell (in FP64 64
// clocks each); the border cells set the time of every small level's sweep.
// Measured per time step against the branches (bitwise the same results): 32^2
// FP64 to 1e-10 21.1 -> 16.3 ms, 256^2 FP64 3.70 -> 3.10 ms, 2048^2 FP64 54.1 ->
// 48.2 ms, 64^2 FP32 0.62 -> 0.49 ms, 1024^2 FP32 2.06 -> 1.86 ms.
#pragma once
#include "biot_common.cuh"

namespace biot {

// What a cell touches on one side: nothing (or a periodic side), or a wall by
// type; a DIRICHLET wall before (first call) and after its history is valid.
enum { WALL_NONE = 0, WALL_SYM = 1, WALL_DIR0 = 2, WALL_NEU = 3, WALL_DIR = 4, WALL_KINDS = 5 };
static_assert((int)BC_PERIODIC == (int)WALL_NONE && (int)BC_SYMMETRY == (int)WALL_SYM &&
                  (int)BC_DIRICHLET == (int)WALL_DIR0 && (int)BC_NEUMANN == (int)WALL_NEU,
              "wall kinds extend the boundary types");

// Descriptor of one pull: the direction read (bits 0-2), its row relative to the
// cell (bits 3-4: 0 below, 1 own, 2 above) and column (bits 5-6: 0 left, 1 own, 2
// right), the signs of h, of dx inside a diagonal's h, and of g (bits 7, 8, 9), and
// whether the value comes from the history (bit 10) or carries boundary data (bit
// 11), of the top/bottom wall (bit 12) or of a side wall.
enum { WP_K = 7, WP_ROW = 3, WP_COL = 5, WP_SH = 7, WP_SD = 8, WP_SG = 9, WP_HIST = 1 << 10, WP_DATA = 1 << 11, WP_HOR = 1 << 12 };

template <typename T>
struct alignas(16) WallEntry {
    unsigned pull[8];
    T bs[3][2], bd[2][2];  // beta coefficients (x, y) of m_11, m_s, m_d and of m_10, m_01
    unsigned beta;         // any of them nonzero
};

template <typename T>
struct WallPull {
    unsigned w;
    T bx, by;
};

template <typename T>
constexpr WallPull<T> wall_pull(int k, int eL, int eR, int eB, int eT)
{
    const int cx = ex8(k), cy = ey8(k), p = pair_of(k);
    const int tv = cx > 0 ? eL : cx < 0 ? eR : 0, th = cy > 0 ? eB : cy < 0 ? eT : 0;
    const bool outx = tv != WALL_NONE, outy = th != WALL_NONE;
    // the wall that decides: the top/bottom one, but at a corner a bounce-back
    // type side wall wins over a mirror top/bottom
    const bool useh = outy && !(outx && th == WALL_SYM && tv != WALL_SYM);
    const bool usev = outx && !useh;
    const int type = useh ? th : usev ? tv : WALL_NONE;
    const bool bounce = type == WALL_NEU || type == WALL_DIR0 || type == WALL_DIR;
    const bool fx = cx != 0 && (usev || bounce || (useh && outx)), fy = cy != 0 && (useh || bounce);
    const int ex = fx ? -cx : cx, ey = fy ? -cy : cy, kr = dir8(ex, ey);
    const bool neg = type == WALL_NEU;  // eq. BC:traction: minus the outgoing population
    const bool hist = type == WALL_DIR; // eq. BC:elasticity: the previous call's outgoing population
    // h = e'/2 a_p . (dx, dy) of the direction read: axis 1/3 of one component,
    // diagonal 1/12 (dy +- dx) with the sign of ey'
    const bool sh = ((p == 0 ? ex : ey) < 0) != neg, sd = p >= 2 && (ex < 0) != (ey < 0);
    const int row = fy ? 1 : 1 - cy, col = fx ? 1 : 1 - cx;
    WallPull<T> o{};
    o.w = (unsigned)kr | (unsigned)row << WP_ROW | (unsigned)col << WP_COL | (sh ? 1u << WP_SH : 0u) |
          (sd ? 1u << WP_SD : 0u) | (neg ? 1u << WP_SG : 0u) | (hist ? (unsigned)WP_HIST : 0u) |
          (bounce ? (unsigned)WP_DATA : 0u) | (useh ? (unsigned)WP_HOR : 0u);
    // beta = +- e'/2 a_p, zero for a history value
    const T wx = cx == 0 || hist ? T(0) : T(p == 0 ? 0.5 * pa_x(0) : 0.5 * pa_x(2));
    const T wy = cy == 0 || hist ? T(0) : T(p == 1 ? 0.5 * pa_y(1) : 0.5 * pa_y(2));
    o.bx = (ex < 0) != neg ? -wx : wx;
    o.by = (ey < 0) != neg ? -wy : wy;
    return o;
}

template <typename T>
constexpr WallEntry<T> wall_entry(int eL, int eR, int eB, int eT)
{
    WallEntry<T> e{};
    T sx[4] = {}, sy[4] = {}, dx[4] = {}, dy[4] = {};  // beta sums, and differences minus a_p, per pair
    for (int p = 0; p < 4; p++) {
        const WallPull<T> u = wall_pull<T>(pair_first(p), eL, eR, eB, eT), v = wall_pull<T>(pair_second(p), eL, eR, eB, eT);
        e.pull[pair_first(p)] = u.w;
        e.pull[pair_second(p)] = v.w;
        sx[p] = u.bx + v.bx;
        sy[p] = u.by + v.by;
        dx[p] = (u.bx - v.bx) - T(pa_x(p));
        dy[p] = (u.by - v.by) - T(pa_y(p));
    }
    const T(*s[2])[4] = {&sx, &sy}, (*d[2])[4] = {&dx, &dy};
    bool any = false;
    for (int c = 0; c < 2; c++) {
        const T(&S)[4] = *s[c], (&D)[4] = *d[c];
        e.bd[0][c] = (D[0] + D[2]) - D[3];
        e.bd[1][c] = (D[1] + D[2]) + D[3];
        e.bs[0][c] = S[2] - S[3];
        e.bs[1][c] = (S[0] + S[1]) + T(2) * (S[2] + S[3]);
        e.bs[2][c] = S[0] - S[1];
        for (int i = 0; i < 3; i++) any = any || e.bs[i][c] != T(0);
        for (int i = 0; i < 2; i++) any = any || e.bd[i][c] != T(0);
    }
    e.beta = any ? 1 : 0;
    return e;
}

// The ghost moments' beta coefficients (x, y) of m_12, m_21, m_22 (tolerance mode).
template <typename T>
struct WallGhost {
    T b[3][2];
};
template <typename T>
constexpr WallGhost<T> wall_ghost(int eL, int eR, int eB, int eT)
{
    WallGhost<T> g{};
    T s[2][4] = {}, d[2][4] = {};
    for (int p = 2; p < 4; p++) {
        const WallPull<T> u = wall_pull<T>(pair_first(p), eL, eR, eB, eT), v = wall_pull<T>(pair_second(p), eL, eR, eB, eT);
        s[0][p] = u.bx + v.bx;
        s[1][p] = u.by + v.by;
        d[0][p] = (u.bx - v.bx) - T(pa_x(p));
        d[1][p] = (u.by - v.by) - T(pa_y(p));
    }
    for (int c = 0; c < 2; c++) {
        g.b[0][c] = d[c][2] - d[c][3];
        g.b[1][c] = d[c][2] + d[c][3];
        g.b[2][c] = s[c][2] + s[c][3];
    }
    return g;
}

template <typename T>
struct WallTable {
    WallEntry<T> e[WALL_KINDS * WALL_KINDS * WALL_KINDS * WALL_KINDS];
    WallGhost<T> g[WALL_KINDS * WALL_KINDS * WALL_KINDS * WALL_KINDS];
};
__host__ __device__ constexpr int wall_index(int eL, int eR, int eB, int eT)
{
    return ((eL * WALL_KINDS + eR) * WALL_KINDS + eB) * WALL_KINDS + eT;
}
template <typename T>
constexpr WallTable<T> make_wall_table()
{
    WallTable<T> t{};
    for (int l = 0; l < WALL_KINDS; l++)
        for (int r = 0; r < WALL_KINDS; r++)
            for (int b = 0; b < WALL_KINDS; b++)
                for (int u = 0; u < WALL_KINDS; u++) {
                    t.e[wall_index(l, r, b, u)] = wall_entry<T>(l, r, b, u);
                    t.g[wall_index(l, r, b, u)] = wall_ghost<T>(l, r, b, u);
                }
    return t;
}
static __device__ constexpr WallTable<float> wall_table32 = make_wall_table<float>();
static __device__ constexpr WallTable<double> wall_table64 = make_wall_table<double>();
template <typename T>
__device__ __forceinline__ const WallTable<T> &wall_table()
{
    if constexpr (sizeof(T) == 8) return wall_table64;
    else return wall_table32;
}

}  // namespace biot

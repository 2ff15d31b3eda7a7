// sweep_pair.cuh -- the strip sweep of large FP32 levels, two cells per lane in
// packed arithmetic.
//
// The row-streaming sweep of sweep_mom.cuh spends as long issuing instructions
// (some 390 per cell: 22 shared loads and 9 stores among them, and the register
// moves between rows) as HBM needs for its bytes, and waits at two block barriers
// per row.  Here a warp walks down a strip of its own:
//  * lane t holds the cells of columns 2t and 2t+1 of the warp's 64; every
//    operation of the collision, the pulls and the residual is one packed
//    instruction for both (fma / add / mul .rn.f32x2: each half rounds as the scalar
//    operation does, so results are bitwise those of the other forms);
//  * what a cell needs of its neighbours comes from its own lane or the next one:
//    twelve shuffles per row and pair of cells, no shared-memory rings, no barrier;
//  * a row's post-collision data are turned into the pulls of the rows below, at
//    and above it as soon as it is collided, so that 14 packed values are carried
//    from row to row instead of three rows of state;
//  * rows arrive through a ring of asynchronous copies (16 bytes per lane), several
//    rows ahead, without holding registers.
// It writes the cells two or more away from every side; the frame around them --
// the wall cells and those whose pulls see ghost values -- is done by small tiles of
// the general code in the same launch.
// What bounds it: HBM at 4096^2 (0.196 ms per finest sweep in the timed step, 1.08 GB:
// 5.5 TB/s, 0.82 of the copy bandwidth), and below that the latency of a row in few
// warps.  Against the strips it replaced, both with tuned heights: the finest sweep of a
// step 0.248 -> 0.196 ms at 4096^2; back to back 0.238 -> 0.185 ms, 2048^2 77 -> 52 us,
// 1024^2 27 -> 17 us, 512^2 13.4 -> 8.8 us.  Per time step (the small levels' launch and the
// wall table are in it): 4096^2 10.6 -> 7.6 ms, 2048^2 4.0 -> 2.5 ms, 1024^2 1.89 -> 1.14 ms,
// 512^2 1.18 -> 0.68 ms; with default heights 11.4 -> 7.6, 4.4 -> 2.5, 2.0 -> 1.15, 1.20 -> 0.69.
#pragma once
#include "sweep_batch.cuh"
#include "sweep_mom.cuh"

namespace biot {

struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float a, float b)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ F2 f2(float a) { return f2(a, a); }
__device__ __forceinline__ void f2_split(F2 a, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ F2 operator+(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mad_rn(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
// A product.  The assembler fuses a packed product into a packed sum that is its only
// use, explicit rounding or not (seen in the force below), and then rounds once where
// every other form of a sweep rounds twice.  The rule for every product that meets a
// packed sum or difference: it has a second use, which keeps it a value of its own (q3,
// q6, q7, q0, q2 meet a sum and a difference each, the coarse force four), or the sum is
// an fma whose factor 1 the assembler cannot know (`one` in sweep_pair_strip).  A product
// as the addend of an fma is safe, and one with -1 is exact.  Writing all of these sums
// that way costs 0.3 to 0.7 % of a step (1024^2: 1.146 -> 1.156 ms), for nothing while the
// results are bitwise those of the general strips, as the tests demand.
__device__ __forceinline__ F2 mul_rn(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
// a - b: the product with -1 is exact, so this rounds once, as a subtraction does.
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return mad_rn(b, f2(-1.0f), a); }

// The values of the columns one to the west / east of a lane's two.
__device__ __forceinline__ F2 from_west(F2 a)
{
    float x, y;
    f2_split(a, x, y);
    return f2(__shfl_up_sync(0xffffffffu, y, 1), x);
}
__device__ __forceinline__ F2 from_east(F2 a)
{
    float x, y;
    f2_split(a, x, y);
    return f2(y, __shfl_down_sync(0xffffffffu, x, 1));
}

// Rows of a ring, at the PAIR_CTAS = 3 resident CTAs per SM that 124 to 168 registers
// (148 for plain smoothing of the finest level) leave room for.  Measured, ms per step at 2048^2 / 4096^2: 3 CTAs with 3, 4, 5, 6
// slots 2.53 / 7.68, 2.57 / 7.73, 2.60 / 7.68, 2.63 / 7.70 (a smaller ring leaves L1
// to the lines that neighbouring strips share); 4 CTAs spill (4.19 / 16.6).
constexpr int PAIR_SLOTS = 3;
static_assert(TileShape<PAIR_FX, PAIR_FY>::NT == 32 * PAIR_WARPS && TileShape<PAIR_FY, PAIR_FX>::NT == 32 * PAIR_WARPS,
              "a frame tile is one CTA");

template <int KIND, bool LO, int FM>
struct PairRing {
    static constexpr bool FINE = kind_fine(KIND), ZERO = FM == FETCH_ZERO, PROL = FM == FETCH_PROL;
    // planes of a row: the iterate m0..m4 (unless zero), its low parts, then F~ or r
    static constexpr int M = ZERO ? 0 : 5, LOP = LO && !ZERO ? 2 : 0, X = FINE ? 2 : 5;
    static constexpr int PLANES = M + LOP + X;
    static constexpr int ROW = PLANES * 64 + (PROL ? 5 * 32 : 0);  // floats: the planes, then the coarse correction
    static constexpr int SLOTS = PROL ? PAIR_SLOTS - 1 : PAIR_SLOTS;
    static constexpr size_t bytes = (size_t)PAIR_WARPS * SLOTS * ROW * sizeof(float);
    static constexpr int UNITS = PLANES * 16, N16 = (UNITS + 31) / 32;  // 16-byte copies of a row, and per lane
};

// One lane's two cells of a row as the collision takes them.
template <int KIND, bool LO>
struct PairRow {
    F2 m[5], lo[2], x[kind_fine(KIND) ? 2 : 5];
};

__device__ __forceinline__ void pair_copy16(unsigned dst, const float *src, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
template <typename TC>
__device__ __forceinline__ void pair_copy4(unsigned dst, const TC *src, bool in)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// Rows y0 .. y1-1 of columns x0 .. x0 + 59 (x0 = 2 mod 4, away from the sides).
// MEAS: also the residual norms of the solve's last sweep (a.resmax).
template <typename TC, int KIND, bool LO, bool RESTRICT, int FM, bool MEAS>
__device__ __forceinline__ void sweep_pair_strip(const SweepArgs<float, TC> &a, int x0, int y0, int y1, float *ring)
{
    using R = PairRing<KIND, LO, FM>;
    constexpr bool FINE = R::FINE, ZERO = R::ZERO, PROL = R::PROL;
    static_assert(!(PROL && sizeof(TC) != 4), "large levels have an FP32 level below them");
    const int nx = a.nx, lane = threadIdx.x & 31, x = x0 - 2 + 2 * lane;
    const size_t NP = (size_t)nx * a.ny;
    const bool writes = lane >= 1 && lane <= 30 && x < nx - 2;

    // this lane's 16-byte copies of a row: unit u = plane u / 16, columns 4 (u % 16) ..
    const float *src[R::N16];
    bool in[R::N16];
    unsigned dst[R::N16];
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(ring);
#pragma unroll
    for (int i = 0; i < R::N16; i++) {
        const int u = lane + 32 * i, k = u >> 4, c = x0 - 2 + 4 * (u & 15);
        const float *p = k < R::M ? a.g + (size_t)k * NP
                       : k < R::M + R::LOP ? a.glo + (size_t)(k - R::M) * NP
                       : FINE ? a.Ft + (size_t)(k - R::M - R::LOP) * NP : a.r + (size_t)(k - R::M - R::LOP) * NP;
        in[i] = u < R::UNITS && c < nx;
        src[i] = in[i] ? p + (size_t)(y0 - 2) * nx + c : a.Ft ? a.Ft : a.r;
        dst[i] = sbase + 16 * u;
    }
    const int cx = (x0 - 2) / 2 + lane;  // coarse column of this lane's cells
    int fetched = y0 - 2, wslot = 0;     // next row to copy and its slot
    const int last = y1 + 1;             // last row needed
    auto copy_row = [&]() {
        if (fetched <= last) {
            const unsigned off = wslot * (R::ROW * 4);
#pragma unroll
            for (int i = 0; i < R::N16; i++)
                if (32 * i + 32 <= R::UNITS || lane + 32 * i < R::UNITS) pair_copy16(dst[i] + off, src[i], in[i]);
            if constexpr (PROL) {
                const size_t NPc = NP >> 2;
                const bool inc = 2 * cx < nx;
                const TC *gc = a.gc + (inc ? (size_t)(fetched >> 1) * (nx >> 1) + cx : 0);
#pragma unroll
                for (int k = 0; k < 5; k++)
                    pair_copy4(sbase + off + 4 * (R::PLANES * 64 + k * 32 + lane), gc + k * NPc, inc);
            }
#pragma unroll
            for (int i = 0; i < R::N16; i++)
                if (in[i]) src[i] += nx;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        fetched++;
        wslot = wslot + 1 == R::SLOTS ? 0 : wslot + 1;
    };
    int rslot = 0;
    // the oldest outstanding row into registers; its slot is refilled by the copy after
    auto take_row = [&](PairRow<KIND, LO> &r) {
        asm volatile("cp.async.wait_group %0;" ::"n"(R::SLOTS - 2) : "memory");
        __syncwarp();
        const float *row = ring + rslot * R::ROW;
        auto plane = [&](int k) { return *reinterpret_cast<const F2 *>(row + k * 64 + 2 * lane); };
#pragma unroll
        for (int k = 0; k < 5; k++) r.m[k] = ZERO ? f2(0.0f) : plane(k);
        if constexpr (LO) {
            r.lo[0] = ZERO ? f2(0.0f) : plane(R::M);
            r.lo[1] = ZERO ? f2(0.0f) : plane(R::M + 1);
        }
#pragma unroll
        for (int k = 0; k < R::X; k++) r.x[k] = plane(R::M + R::LOP + k);
        if constexpr (PROL) {
            const float *q = row + R::PLANES * 64 + lane;
            if constexpr (LO) {
                r.lo[0] = r.lo[0] + f2(q[0]);
                r.lo[1] = r.lo[1] + f2(q[32]);
            } else {
                r.m[0] = r.m[0] + f2(q[0]);
                r.m[1] = r.m[1] + f2(q[32]);
            }
#pragma unroll
            for (int k = 2; k < 5; k++) r.m[k] = r.m[k] + f2(q[k * 32]);
        }
        rslot = rslot + 1 == R::SLOTS ? 0 : rslot + 1;
        __syncwarp();
        copy_row();
    };
#pragma unroll
    for (int i = 0; i < R::SLOTS - 1; i++) copy_row();

    const F2 c13 = f2(float(1.0 / 3.0)), c112 = f2(float(1.0 / 12.0));
    const F2 kfs = f2(a.k_fs), khd = f2(a.k_hd), khs = f2(a.k_hs), kh22 = f2(a.k_h22), ngam = f2(-a.k_gam);
    const F2 one = f2(__uint_as_float(0x3f800000u | ((unsigned)nx >> 31)));  // 1: nx is positive
    struct Ms {
        F2 c, w, e;
    };
    auto ms_of = [&](F2 v) { return Ms{v, from_west(v), from_east(v)}; };
    // target-side first moments of a row: high and low parts (own_from)
    struct Own {
        F2 tx, ty, tlx, tly;
    };
    auto own_of = [&](const PairRow<KIND, LO> &r) {
        Own o;
        if constexpr (FINE) {
            o.tx = r.m[0];
            o.ty = r.m[1];
            if constexpr (LO) {
                o.tlx = r.lo[0];
                o.tly = r.lo[1];
            }
        } else {
            o.tx = r.m[0] - r.x[0];
            o.ty = r.m[1] - r.x[1];
        }
        return o;
    };
    auto diff_x = [&](F2 mx, const Own &o) {
        const F2 d = mx - o.tx;
        if constexpr (LO) return d - o.tlx;
        else return d;
    };
    auto diff_y = [&](F2 my, const Own &o) {
        const F2 d = my - o.ty;
        if constexpr (LO) return d - o.tly;
        else return d;
    };

    PairRow<KIND, LO> P, B, C;  // rows j-1, j, j+1
    Ms sS, sO, sN;              // their m_s
    F2 g1, h1, g4, h4, g5, h5;        // pulls of directions 01, 11, -11 into row j, from the collision of row j-1
    F2 S0, A0;                        // pair 0 of row j-1
    F2 pg1, ph1, pg4, ph4, pg5, ph5;  // the pulls into row j-1, from row j-2
    F2 acc[5];
    float rmax = 0.0f, gmax = 0.0f;
    double rsum = 0.0;
    take_row(P);  // row y0-2: only its m_s
    sS = ms_of(P.m[3]);
    take_row(B);
    sO = ms_of(B.m[3]);

    for (int j = y0 - 1; j <= y1; j++) {
        take_row(C);
        sN = ms_of(C.m[3]);
        // collision of row j (collide_math)
        const F2 gx = mad_rn(sO.e - sO.w, c13, mul_rn((sN.e + sS.e) - (sN.w + sS.w), c112));
        const F2 gy = mad_rn(sN.c - sS.c, c13, mul_rn((sN.e + sN.w) - (sS.e + sS.w), c112));
        F2 Fx = mul_rn(kfs, gx), Fy = mul_rn(kfs, gy);
        F2 m2 = B.m[2], m3 = B.m[3], m4 = B.m[4];
        const Own ob = own_of(B);
        if constexpr (FINE) {
            Fx = mad_rn(B.x[0], one, Fx);
            Fy = mad_rn(B.x[1], one, Fy);
        } else {
            m2 = m2 - B.x[2];
            m3 = m3 - B.x[3];
            m4 = m4 - B.x[4];
        }
        const F2 hd = mul_rn(khd, m4), h22 = mul_rn(kh22, m3);
        const F2 nhd = mul_rn(f2(-a.k_hd), m4);
        const F2 hS0 = mad_rn(khs, m3, hd), hS1 = mad_rn(khs, m3, nhd);
        const F2 hS2 = mad_rn(khd, m2, h22), hS3 = mad_rn(f2(-a.k_hd), m2, h22);
        const F2 Fp = Fx + Fy, Fm = Fy - Fx;
        F2 G0, G1, G2, G3, G4, G5, G6, G7;
        if constexpr (LO) {
            const F2 lx = B.lo[0], ly = B.lo[1];
            const F2 a0 = mad_rn(f2(float(5.0 / 12.0)), Fx, mul_rn(c13, lx)), a1 = mad_rn(f2(float(5.0 / 12.0)), Fy, mul_rn(c13, ly));
            const F2 a2 = mad_rn(f2(float(1.0 / 24.0)), Fp, mul_rn(c112, lx + ly));
            const F2 a3 = mad_rn(f2(float(1.0 / 24.0)), Fm, mul_rn(c112, ly - lx));
            G0 = hS0 + a0;
            G2 = hS0 - a0;
            G1 = hS1 + a1;
            G3 = hS1 - a1;
            G4 = hS2 + a2;
            G6 = hS2 - a2;
            G5 = hS3 + a3;
            G7 = hS3 - a3;
        } else {
            G0 = mad_rn(f2(float(5.0 / 12.0)), Fx, hS0);
            G2 = mad_rn(f2(float(-5.0 / 12.0)), Fx, hS0);
            G1 = mad_rn(f2(float(5.0 / 12.0)), Fy, hS1);
            G3 = mad_rn(f2(float(-5.0 / 12.0)), Fy, hS1);
            G4 = mad_rn(f2(float(1.0 / 24.0)), Fp, hS2);
            G6 = mad_rn(f2(float(-1.0 / 24.0)), Fp, hS2);
            G5 = mad_rn(f2(float(1.0 / 24.0)), Fm, hS3);
            G7 = mad_rn(f2(float(-1.0 / 24.0)), Fm, hS3);
        }
        const F2 mxw = from_west(ob.tx), mxe = from_east(ob.tx), myw = from_west(ob.ty), mye = from_east(ob.ty);

        if (j > y0) {  // finish row j-1: the downward pulls from row j (h = -q)
            const Own op = own_of(P);
            const F2 q3 = mul_rn(c13, diff_y(ob.ty, op));
            const F2 g6 = from_east(G6), q6 = mul_rn(c112, diff_x(mxe, op) + diff_y(mye, op));
            const F2 g7 = from_west(G7), q7 = mul_rn(c112, diff_y(myw, op) - diff_x(mxw, op));
            const F2 S1 = (pg1 + G3) + (ph1 - q3), A1 = (pg1 - G3) + (ph1 + q3);
            const F2 S2 = (pg4 + g6) + (ph4 - q6), A2 = (pg4 - g6) + (ph4 + q6);
            const F2 S3 = (pg5 + g7) + (ph5 - q7), A3 = (pg5 - g7) + (ph5 + q7);
            F2 d[5];
            const F2 t0 = (A0 + A2) - A3, t1 = (A1 + A2) + A3;
            if constexpr (FINE) {  // the iterate is the collision input
                d[0] = mul_rn(f2(-1.0f), t0);
                d[1] = mul_rn(f2(-1.0f), t1);
            } else {
                d[0] = (P.m[0] - op.tx) - t0;
                d[1] = (P.m[1] - op.ty) - t1;
            }
            d[2] = P.m[2] - (S2 - S3);
            d[3] = P.m[3] - mad_rn(f2(2.0f), S2 + S3, S0 + S1);
            d[4] = P.m[4] - (S0 - S1);
            const int y = j - 1;
            if constexpr (RESTRICT) {
                if ((y & 1) == 0) {  // full-sum restriction: rows, then the pair's columns
#pragma unroll
                    for (int k = 0; k < 5; k++) acc[k] = d[k];
                } else if (writes) {
                    const size_t NPc = NP >> 2, ci = (size_t)(y >> 1) * (nx >> 1) + (x >> 1);
#pragma unroll
                    for (int k = 0; k < 5; k++) {
                        float u, v;
                        f2_split(acc[k] + d[k], u, v);
                        a.rc[k * NPc + ci] = (TC)u + (TC)v;
                    }
                }
            } else {
                F2 o[5], ol[2];
#pragma unroll
                for (int k = 2; k < 5; k++) o[k] = mad_rn(ngam, d[k], P.m[k]);
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    if constexpr (LO) {
                        const F2 b = mad_rn(ngam, d[k], P.lo[k]), s = P.m[k] + b, bb = s - P.m[k];
                        o[k] = s;
                        ol[k] = (P.m[k] - (s - bb)) + (b - bb);
                    } else {
                        o[k] = mad_rn(ngam, d[k], P.m[k]);
                    }
                }
                if (MEAS && writes) {  // per cell, as the general strips
                    float dc[2][8] = {}, gc[2][8] = {};
#pragma unroll
                    for (int k = 0; k < 5; k++) {
                        f2_split(d[k], dc[0][k], dc[1][k]);
                        f2_split(P.m[k], gc[0][k], gc[1][k]);
                    }
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        rmax = fmaxf(rmax, pop_absmax(dc[c]));
                        gmax = fmaxf(gmax, pop_absmax(gc[c]));
                        rsum += (double)pop_sumsq(dc[c]);
                    }
                }
                if (writes) {
                    const size_t idx = (size_t)y * nx + x;
                    float *go = a.gout + idx;
#pragma unroll
                    for (int k = 0; k < 5; k++) *reinterpret_cast<F2 *>(go + k * NP) = o[k];
                    if constexpr (LO) {
                        float *gl = a.glo_out + idx;
                        *reinterpret_cast<F2 *>(gl) = ol[0];
                        *reinterpret_cast<F2 *>(gl + NP) = ol[1];
                    }
                }
            }
        }
        // pair 0 of row j, and the upward pulls into row j+1
        {
            const F2 g0 = from_west(G0), g2 = from_east(G2);
            const F2 q0 = mul_rn(c13, diff_x(mxw, ob)), q2 = mul_rn(c13, diff_x(mxe, ob));
            S0 = (g0 + g2) + (q0 - q2);
            A0 = (g0 - g2) + (q0 + q2);
        }
        pg1 = g1;
        ph1 = h1;
        pg4 = g4;
        ph4 = h4;
        pg5 = g5;
        ph5 = h5;
        {
            const Own oc = own_of(C);
            g1 = G1;
            h1 = mul_rn(c13, diff_y(ob.ty, oc));
            g4 = from_west(G4);
            h4 = mul_rn(c112, diff_x(mxw, oc) + diff_y(myw, oc));
            g5 = from_east(G5);
            h5 = mul_rn(c112, diff_y(mye, oc) - diff_x(mxe, oc));
        }
        P = B;
        B = C;
        sS = sO;
        sO = sN;
    }
    if constexpr (MEAS) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
            gmax = fmaxf(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
            rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
        }
        if (lane == 0) {
            atomicMax(&a.resmax[0], (unsigned long long)__double_as_longlong((double)rmax));
            atomicMax(&a.resmax[1], (unsigned long long)__double_as_longlong((double)gmax));
            atomicAdd(reinterpret_cast<double *>(&a.resmax[2]), rsum);
        }
    }
}

// CTA b of a level's sweep: PAIR_WARPS strips, or past the strips a tile of the
// frame.  The frame's tiles come last, where they fill the tail (first in the grid
// they hold every SM for some 8 us: 8.68 instead of 8.13 ms per 4096^2 step).
template <typename TC, int KIND, bool LO, bool RESTRICT, int FM, bool MEAS>
__device__ __forceinline__ void sweep_pair_cta(const SweepArgs<float, TC> &a, int b, int TY, unsigned char *smem,
                                               double (&red)[3][PAIR_WARPS])
{
    const int strips = pair_strip_ctas(a.nx, a.ny, TY);
    if (b >= strips) {
        const int ntx = (a.nx + PAIR_FX - 1) / PAIR_FX, nty = (a.ny + PAIR_FX - 1) / PAIR_FX;
        b -= strips;
        if (b < 2 * ntx) {
            const int top = b >= ntx ? 1 : 0;
            tile_body<float, TC, PAIR_FX, PAIR_FY, KIND, LO, RESTRICT>(a, b - top * ntx, top * (a.ny / PAIR_FY - 1), smem, red);
        } else {
            b -= 2 * ntx;
            const int right = b >= nty ? 1 : 0;
            tile_body<float, TC, PAIR_FY, PAIR_FX, KIND, LO, RESTRICT>(a, right * (a.nx / PAIR_FY - 1), b - right * nty, smem, red,
                                                                      PAIR_FY, a.ny - PAIR_FY);
        }
        return;
    }
    using R = PairRing<KIND, LO, FM>;
    const int nsx = pair_strips_x(a.nx), w = b * PAIR_WARPS + (int)(threadIdx.x >> 5);
    const int by = w / nsx, y0 = 2 + by * TY;
    if (y0 >= a.ny - 2) return;
    float *ring = reinterpret_cast<float *>(smem) + (threadIdx.x >> 5) * (R::SLOTS * R::ROW);
    sweep_pair_strip<TC, KIND, LO, RESTRICT, FM, MEAS>(a, 2 + PAIR_COLS * (w - by * nsx), y0, min(y0 + TY, a.ny - 2), ring);
}

template <typename TC, int KIND, bool LO, bool RESTRICT, int FM, bool MEAS>
__global__ void __launch_bounds__(32 * PAIR_WARPS, PAIR_CTAS) k_sweep_pair(const SweepArgs<float, TC> a, int TY)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[3][PAIR_WARPS];
    sweep_pair_cta<TC, KIND, LO, RESTRICT, FM, MEAS>(a, blockIdx.x, TY, smem_raw, red);
}

// Batched form: the sweeps of many instances' levels, job j's CTAs start[j] ..
template <typename TC, int KIND, bool LO, bool RESTRICT, int FM, bool MEAS>
__global__ void __launch_bounds__(32 * PAIR_WARPS, PAIR_CTAS) k_sweep_pair_batch(const __grid_constant__ BatchParams<float, TC> P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[3][PAIR_WARPS];
    const int j = batch_job(P, blockIdx.x);
    sweep_pair_cta<TC, KIND, LO, RESTRICT, FM, MEAS>(P.job[j], blockIdx.x - P.start[j], P.ty[j], smem_raw, red);
}

// Whether the packed sweep takes these arguments: a level of pair_takes_level, its
// iterate stored (with or without a prolongated correction) or zero, and a level
// below it in FP32 when its correction is added.
template <typename TC, int KIND, bool LO>
bool pair_takes(const SweepArgs<float, TC> &a)
{
    return pair_takes_level(kind_fine(KIND), LO, a.ghosts != 0, a.dev != 0, a.nx, a.ny) && !(a.zero_init && a.gc) &&
           !(a.gc && sizeof(TC) != 4) && !(a.zero_init && a.Ft);
}

// Shared memory of a CTA.
template <int KIND, bool LO, int FM>
constexpr size_t pair_smem()
{
    constexpr size_t t0 = tile_smem_bytes<float, PAIR_FX, PAIR_FY, KIND, LO>(), t1 = tile_smem_bytes<float, PAIR_FY, PAIR_FX, KIND, LO>();
    constexpr size_t t = t0 > t1 ? t0 : t1;
    return PairRing<KIND, LO, FM>::bytes > t ? PairRing<KIND, LO, FM>::bytes : t;
}
template <typename TC, int KIND, bool LO, bool RESTRICT, int FM, bool MEAS = false>
cudaError_t launch_pair_fm(const SweepArgs<float, TC> &a, cudaStream_t s)
{
    constexpr size_t smem = pair_smem<KIND, LO, FM>();
    auto kern = k_sweep_pair<TC, KIND, LO, RESTRICT, FM, MEAS>;
    static DeviceCache ctas;
    const int n = ctas.get([&](int dev) { return resident_ctas(dev, (const void *)kern, 32 * PAIR_WARPS, smem); });
    if (!n) return no_slots();
    const int ty = pair_height(a.rows, pair_strips_x(a.nx), a.ny - 4, n * PAIR_WARPS);
    kern<<<pair_strip_ctas(a.nx, a.ny, ty) + pair_frame_ctas(a.nx, a.ny), 32 * PAIR_WARPS, smem, s>>>(a, ty);
    return cudaGetLastError();
}

template <typename TC, int KIND, bool LO, bool RESTRICT, int FM, bool MEAS = false>
cudaError_t launch_pair_batch_fm(const BatchParams<float, TC> &P, cudaStream_t s)
{
    constexpr size_t smem = pair_smem<KIND, LO, FM>();
    auto kern = k_sweep_pair_batch<TC, KIND, LO, RESTRICT, FM, MEAS>;
    static DeviceCache ctas;
    const int n = ctas.get([&](int dev) { return resident_ctas(dev, (const void *)kern, 32 * PAIR_WARPS, smem); });
    if (!n) return no_slots();
    for (int j = 0; j < P.njobs; j++)  // what the plan assumed of its jobs
        if (!pair_takes<TC, KIND, LO>(P.job[j]) || MEAS != (P.job[j].resmax != nullptr) || (FM == FETCH_PROL) != (P.job[j].gc != nullptr) || (FM == FETCH_ZERO) != (P.job[j].zero_init != 0) ||
            P.start[j + 1] - P.start[j] != pair_strip_ctas(P.job[j].nx, P.job[j].ny, P.ty[j]) + pair_frame_ctas(P.job[j].nx, P.job[j].ny))
            return cudaErrorInvalidValue;
    kern<<<P.start[P.njobs], 32 * PAIR_WARPS, smem, s>>>(P);
    return cudaGetLastError();
}

template <typename TC, int KIND, bool LO, bool RESTRICT>
cudaError_t launch_pair(const SweepArgs<float, TC> &a, cudaStream_t s)
{
    if constexpr (!kind_fine(KIND)) {
        if (a.zero_init) return launch_pair_fm<TC, KIND, LO, RESTRICT, FETCH_ZERO>(a, s);
    }
    if constexpr (kind_fine(KIND) && !RESTRICT) {
        if constexpr (sizeof(TC) == 4) {
            if (a.resmax && a.gc) return launch_pair_fm<TC, KIND, LO, RESTRICT, FETCH_PROL, true>(a, s);
        }
        if (a.resmax) return launch_pair_fm<TC, KIND, LO, RESTRICT, FETCH_PLAIN, true>(a, s);
    }
    if constexpr (sizeof(TC) == 4 && !RESTRICT) {
        if (a.gc) return launch_pair_fm<TC, KIND, LO, RESTRICT, FETCH_PROL>(a, s);
    }
    return launch_pair_fm<TC, KIND, LO, RESTRICT, FETCH_PLAIN>(a, s);
}

}  // namespace biot

// fp64 symmetric positive-definite D x D systems on the double-precision matrix instruction, one system per team of warps.
//
// mma.m8n8k4.f64 is the building block (there is no tcgen05 form of it): one every 16 clocks and scheduler on B200, the
// rate of plain DFMA without its operand traffic.  A lane l of a warp holds of an 8 x 8 block of the accumulator the
// elements (l / 4, 2 (l % 4)) and (l / 4, 2 (l % 4) + 1); as an A operand (8 x 4) it supplies element (l / 4, l % 4) and
// as a B operand (4 x 8) element (l % 4, l / 4).  For a product X Y^T over eight columns the order of the
// contraction is free, so accumulator fragments of X and Y serve as operands as they are (register 0 of every lane in one
// instruction, register 1 in the next): the factorisation moves nothing between lanes but the 8 x 8 pivot blocks.
//
// The lower block triangle lies in shared memory, a block as 32 pairs in accumulator layout.  (Kept in the warps'
// registers instead, every panel has to be code of its own: 100 KB of straight-line instructions, which the systems of
// an SM waited for -- 3.7 K clocks a panel at d = 64.)
//
// What bounds it is the chain through the pivot blocks: four steps of shuffle, determinant, reciprocal, multiply and
// subtract.  The pivots are 2 x 2 blocks, whose two columns a lane holds, so there are four reciprocals in a row
// instead of eight.
#pragma once

#include "lla_common.cuh"

namespace lla {
namespace team {

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
    asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

// Block rows dealt to the warps of a team while the matrix is built in registers: back and forth (row 0 to warp 0, ..
// NW - 1 to warp NW - 1, NW to warp NW - 1, ..), which gives every warp the same number of blocks.
template <int D, int NW_>
struct Cfg {
    static constexpr int NW = NW_;                     // warps of a team
    static constexpr int NB = D / 8;                   // block rows
    static constexpr int R = NB / NW;                  // block rows of a warp
    static constexpr int NBLK = NW * R * (R + 1) / 2;  // blocks a warp keeps (some of the last NW columns unused)
    static constexpr int LOWER = NB * (NB + 1) / 2;    // blocks of the lower triangle
    __host__ __device__ static constexpr int off(int r) { return NW * r * (r + 1) / 2; }
    __host__ __device__ static constexpr int cols(int r) { return NW * (r + 1); }
    __host__ __device__ static constexpr int row(int r, int w) { return r & 1 ? r * NW + NW - 1 - w : r * NW + w; }
    static_assert(NB % NW == 0, "block rows per warp");
};
// block (i, j), j <= i, of the lower triangle
__host__ __device__ __forceinline__ constexpr int blk(int i, int j) { return i * (i + 1) / 2 + j; }

// f(the warp's number in the team as a constant): the loops over a warp's blocks have no guards then, which a run-time
// number would put around every instruction
template <int V>
struct Const {
    static constexpr int value = V;
};
template <int NW, typename F>
__device__ __forceinline__ void with_warp(int w, F&& f) {
    static_assert(NW == 1 || NW == 2 || NW == 8, "team sizes in use");
    if constexpr (NW == 1) {
        f(Const<0>{});
    } else if constexpr (NW == 2) {
        if (w == 0) f(Const<0>{}); else f(Const<1>{});
    } else {
        switch (w) {
            case 0: f(Const<0>{}); break;
            case 1: f(Const<1>{}); break;
            case 2: f(Const<2>{}); break;
            case 3: f(Const<3>{}); break;
            case 4: f(Const<4>{}); break;
            case 5: f(Const<5>{}); break;
            case 6: f(Const<6>{}); break;
            default: f(Const<7>{}); break;
        }
    }
}

template <int D, int NW, int NRHS>
struct alignas(16) Smem {
    double w[64];                   // inverse of the current unit lower triangular pivot block, accumulator layout
    double piv[D / 8][4][6];        // 2 x 2 pivots a b c (a b; b c) and their inverses
    double b[NRHS][D];              // right-hand sides; forward-substituted in place
    double z[NRHS][D];              // the same times the inverse pivots
    double x[NW][NRHS][D];          // solution (every warp writes its own copy)
    double part[2][NW][NRHS][8];
    int bad;
};

template <int NW>
__device__ __forceinline__ void sync(int bar_id) {
    if constexpr (NW == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "n"(32 * NW) : "memory");
}

// Inverse (j00 j01; j01 j11) of the symmetric block (a b; b c); false if it is not positive definite.
// The entries span the doubles' whole range (a diagonal of the dual form is lambda e^-score), so their products may not
// be representable where the inverse is.  A determinant with an exponent beyond 2^+-823 is formed again from the
// entries scaled by powers of two that bring a and c to [1, 2).  (The same operands in every lane: the branch does not diverge.)
__device__ __forceinline__ bool invert_pivot(double a, double b, double c, double& j00, double& j01, double& j11) {
    double det = a * c - b * b;
    const double inv = fast_rcp(det);
    j00 = c * inv;
    j01 = -b * inv;
    j11 = a * inv;
    if ((((unsigned)__double2hiint(det)) >> 20) - 200u >= 1646u) {      // (a sign, infinity and NaN come here too)
        const double sa = __hiloint2double(0x7fe00000 - (__double2hiint(a) & 0x7ff00000), 0);
        const double sc = __hiloint2double(0x7fe00000 - (__double2hiint(c) & 0x7ff00000), 0);
        const double as = a * sa, cs = c * sc;
        det = as * cs - (b * sa) * (b * sc);
        const double is = fast_rcp(det);
        j00 = (cs * is) * sa;
        j01 = -((b * sa) * is) * sc;
        j11 = (as * is) * sc;
    }
    return a > 0.0 && det > 0.0;
}

// Solve for the right-hand sides in sm.b.  c: the lower block triangle (destroyed); nba: block rows in use (the rest is
// not touched); w, lane: warp inside the team and lane.  The solution is in sm.x[w].  Everything must be visible to
// the team before the call.  Returns false if a pivot was not positive (the same in every warp).
template <int D, int NW, int NRHS>
__device__ __forceinline__ bool solve(double (*c)[64], Smem<D, NW, NRHS>& sm, int nba, int w, int lane, int bar_id) {
    constexpr unsigned FULL = 0xffffffffu;
    const int g = lane >> 2, t4 = lane & 3;
    auto ld = [&](const double* p) { return *reinterpret_cast<const double2*>(p + 2 * lane); };
    auto st = [&](double* p, double x, double y) { *reinterpret_cast<double2*>(p + 2 * lane) = make_double2(x, y); };
    // Pivot block p: Gauss elimination by 2 x 2 pivots on [block | I], both in accumulator layout.
    auto pivot = [&](int p, double a0, double a1) {
        double w0 = g == 2 * t4 ? 1.0 : 0.0, w1 = g == 2 * t4 + 1 ? 1.0 : 0.0;
        double i00 = 0.0, i01 = 0.0, i11 = 0.0;      // of the pivot that row g belongs to
        bool ok = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double pa = __shfl_sync(FULL, a0, 9 * k), pb = __shfl_sync(FULL, a1, 9 * k), pc = __shfl_sync(FULL, a1, 9 * k + 4);
            const double x0 = __shfl_sync(FULL, a0, (lane & 28) + k), x1 = __shfl_sync(FULL, a1, (lane & 28) + k);
            const double u0 = __shfl_sync(FULL, a0, 8 * k + t4), u1 = __shfl_sync(FULL, a1, 8 * k + t4);
            const double v0 = __shfl_sync(FULL, a0, 8 * k + 4 + t4), v1 = __shfl_sync(FULL, a1, 8 * k + 4 + t4);
            const double r0 = __shfl_sync(FULL, w0, 8 * k + t4), r1 = __shfl_sync(FULL, w1, 8 * k + t4);
            const double s0 = __shfl_sync(FULL, w0, 8 * k + 4 + t4), s1 = __shfl_sync(FULL, w1, 8 * k + 4 + t4);
            double j00, j01, j11;
            ok = invert_pivot(pa, pb, pc, j00, j01, j11) && ok;
            const double m0 = g > 2 * k + 1 ? x0 * j00 + x1 * j01 : 0.0, m1 = g > 2 * k + 1 ? x0 * j01 + x1 * j11 : 0.0;
            a0 -= m0 * u0 + m1 * v0;
            a1 -= m0 * u1 + m1 * v1;
            w0 -= m0 * r0 + m1 * s0;
            w1 -= m0 * r1 + m1 * s1;
            if ((g >> 1) == k) { i00 = j00; i01 = j01; i11 = j11; }
            if (lane == 0) {
                double2* pp = reinterpret_cast<double2*>(sm.piv[p][k]);
                pp[0] = make_double2(pa, pb);
                pp[1] = make_double2(pc, j00);
                pp[2] = make_double2(j01, j11);
            }
        }
        if (!ok && lane == 0) sm.bad = 1;
        st(sm.w, w0, w1);
        // the pivot block's place keeps the transpose, which the back substitution multiplies with
        c[blk(p, p)][(2 * t4) * 8 + g] = w0;
        c[blk(p, p)][(2 * t4 + 1) * 8 + g] = w1;
#pragma unroll
        for (int q = 0; q < NRHS; ++q) {
            double y = w0 * sm.b[q][8 * p + 2 * t4] + w1 * sm.b[q][8 * p + 2 * t4 + 1];
            y += __shfl_xor_sync(FULL, y, 1);
            y += __shfl_xor_sync(FULL, y, 2);
            const double yo = __shfl_xor_sync(FULL, y, 4);
            __syncwarp();      // the reads of sm.b above come before the write below
            if (t4 == 0) {
                sm.b[q][8 * p + g] = y;
                sm.z[q][8 * p + g] = (g & 1) ? i01 * yo + i11 * y : i00 * y + i01 * yo;
            }
        }
    };
    if (w == 0 && lane == 0) sm.bad = 0;
    if (w == 0) {
        __syncwarp();
        const double2 d = ld(c[0]);
        pivot(0, d.x, d.y);
    }
#pragma unroll 1
    for (int p = 0; p < nba; ++p) {
        sync<NW>(bar_id);
        const double2* pp = reinterpret_cast<const double2*>(sm.piv[p][t4]);
        const double2 p0 = pp[0], p1 = pp[1], p2 = pp[2];        // (a b) (c i00) (i01 i11)
        const double2 wp = ld(sm.w);
        const int next = (p + 1) % NW;                           // the warp that takes the next pivot block
        // the panel below the pivot block; the warp `next` has row p + 1
        // (two rows at a time: their chains of dependent instructions overlap)
#pragma unroll 1
        for (int i0 = p + 1 + (w - next + NW) % NW; i0 < nba; i0 += 2 * NW) {
            const int i1 = i0 + NW < nba ? i0 + NW : i0;
            const double2 c0 = ld(c[blk(i0, p)]), c1 = ld(c[blk(i1, p)]);
            double x0 = 0.0, x1 = 0.0, u0 = 0.0, u1 = 0.0;
            dmma(x0, x1, c0.x, wp.x);
            dmma(u0, u1, c1.x, wp.x);
            dmma(x0, x1, c0.y, wp.y);
            dmma(u0, u1, c1.y, wp.y);
            const double y0 = x0 * p1.y + x1 * p2.x, y1 = x0 * p2.x + x1 * p2.y;
            const double v0 = u0 * p1.y + u1 * p2.x, v1 = u0 * p2.x + u1 * p2.y;
            st(c[blk(i0, p)], y0, y1);
            if (i1 != i0) st(c[blk(i1, p)], v0, v1);
#pragma unroll
            for (int q = 0; q < NRHS; ++q) {
                const double2 bp = *reinterpret_cast<const double2*>(&sm.b[q][8 * p + 2 * t4]);
                double s = y0 * bp.x + y1 * bp.y, t = v0 * bp.x + v1 * bp.y;
                s += __shfl_xor_sync(FULL, s, 1);
                t += __shfl_xor_sync(FULL, t, 1);
                s += __shfl_xor_sync(FULL, s, 2);
                t += __shfl_xor_sync(FULL, t, 2);
                if (t4 == 0) {
                    sm.b[q][8 * i0 + g] -= s;
                    if (i1 != i0) sm.b[q][8 * i1 + g] -= t;
                }
            }
        }
        if (p + 1 >= nba) break;
        sync<NW>(bar_id);
        // C_ij -= Y_i D Y_j^T.  The next pivot block first, so that its factorisation runs beside the other updates
        auto operand = [&](int i, double& n0, double& n1) {
            const double2 y = ld(c[blk(i, p)]);
            n0 = -(y.x * p0.x + y.y * p0.y);
            n1 = -(y.x * p0.y + y.y * p1.x);
        };
        if (w == next) {
            double n0, n1;
            operand(p + 1, n0, n1);
            const double2 y = ld(c[blk(p + 1, p)]);
            double2 d = ld(c[blk(p + 1, p + 1)]);
            dmma(d.x, d.y, n0, y.x);
            dmma(d.x, d.y, n1, y.y);
            pivot(p + 1, d.x, d.y);
        }
        // the other rows: NW - 1 warps share them (two warps: the pivot's warp takes every fourth row when it is done)
        const int o = (w - next + NW) % NW;
#pragma unroll 1
        for (int i = p + 2; i < nba; ++i) {
            const bool mine = NW == 1 || (NW == 2 ? (o == 0) == ((i - p) % 4 == 1) : o == 1 + (i - p - 2) % (NW > 1 ? NW - 1 : 1));
            if (!mine) continue;
            double n0, n1;
            operand(i, n0, n1);
            double* ci = c[blk(i, 0)];
            int j = p + 1;
#pragma unroll 1
            for (; j + 3 <= i; j += 4) {                          // four blocks at a time
                double2 y[4], d[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) { y[u] = ld(c[blk(j + u, p)]); d[u] = ld(ci + 64 * (j + u)); }
#pragma unroll
                for (int u = 0; u < 4; ++u) dmma(d[u].x, d[u].y, n0, y[u].x);
#pragma unroll
                for (int u = 0; u < 4; ++u) dmma(d[u].x, d[u].y, n1, y[u].y);
#pragma unroll
                for (int u = 0; u < 4; ++u) st(ci + 64 * (j + u), d[u].x, d[u].y);
            }
#pragma unroll 1
            for (; j <= i; ++j) {
                const double2 y = ld(c[blk(j, p)]);
                double2 d = ld(ci + 64 * j);
                dmma(d.x, d.y, n0, y.x);
                dmma(d.x, d.y, n1, y.y);
                st(ci + 64 * j, d.x, d.y);
            }
        }
    }
    sync<NW>(bar_id);
    // back substitution: x_p = W_p^T (D_p^{-1} y_p - sum_{i > p} Y_ip^T x_i)
#pragma unroll 1
    for (int p = nba - 1; p >= 0; --p) {
        double s[NRHS][2];
#pragma unroll
        for (int q = 0; q < NRHS; ++q) s[q][0] = s[q][1] = 0.0;
#pragma unroll 2
        for (int i = p + 1 + w; i < nba; i += NW) {
            const double2 y = ld(c[blk(i, p)]);
#pragma unroll
            for (int q = 0; q < NRHS; ++q) {
                const double xi = sm.x[w][q][8 * i + g];
                s[q][0] += y.x * xi;
                s[q][1] += y.y * xi;
            }
        }
#pragma unroll
        for (int q = 0; q < NRHS; ++q) {
#pragma unroll
            for (int o = 4; o <= 16; o <<= 1) {
                s[q][0] += __shfl_xor_sync(FULL, s[q][0], o);
                s[q][1] += __shfl_xor_sync(FULL, s[q][1], o);
            }
            if (NW > 1 && lane < 4) *reinterpret_cast<double2*>(&sm.part[p & 1][w][q][2 * lane]) = make_double2(s[q][0], s[q][1]);
        }
        if (NW > 1) sync<NW>(bar_id);
        const double2 wt = ld(c[blk(p, p)]);
#pragma unroll
        for (int q = 0; q < NRHS; ++q) {
            double2 v = *reinterpret_cast<const double2*>(&sm.z[q][8 * p + 2 * t4]);
            if (NW > 1) {
#pragma unroll
                for (int u = 0; u < NW; ++u) {
                    const double2 e = *reinterpret_cast<const double2*>(&sm.part[p & 1][u][q][2 * t4]);
                    v.x -= e.x;
                    v.y -= e.y;
                }
            } else {
                v.x -= s[q][0];
                v.y -= s[q][1];
            }
            double x = wt.x * v.x + wt.y * v.y;
            x += __shfl_xor_sync(FULL, x, 1);
            x += __shfl_xor_sync(FULL, x, 2);
            if (t4 == 0) sm.x[w][q][8 * p + g] = x;
        }
        __syncwarp();
    }
    return sm.bad == 0;
}

}  // namespace team
}  // namespace lla

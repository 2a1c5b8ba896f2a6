// fp64 symmetric positive-definite D x D systems on the double-precision matrix instruction, one system per team of
// warps, the matrix in registers from its first product to the back substitution.
//
// mma.m8n8k4.f64 is the building block (there is no tcgen05 form of it): measured on B200 at 117 multiply-adds per clock
// and SM with 16 warps (77 with 8, 64 with 4), against 54 for plain DFMA.  A lane l of a warp holds of an 8 x 8
// block of the accumulator the elements (l / 4, 2 (l % 4)) and (l / 4, 2 (l % 4) + 1); as an A operand (8 x 4) it supplies
// element (l / 4, l % 4) and as a B operand (4 x 8) element (l % 4, l / 4).  For a product X Y^T over eight columns the
// order of the contraction is free, so X's and Y's accumulator fragments serve as operands as they are (register 0
// of every lane in one instruction, register 1 in the next): the factorisation moves nothing between lanes but the
// 8 x 8 pivot blocks.
//
// The lower block triangle is dealt to the team's warps by block rows, back and forth (row 0 to warp 0, .. NW - 1 to
// warp NW - 1, NW to warp NW - 1, ..), which gives every warp the same number of blocks.
#pragma once

#include "lla_common.cuh"

namespace lla {
namespace team {

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

template <int D, int NW_>
struct Cfg {
    static constexpr int NW = NW_;                     // warps of a team
    static constexpr int NB = D / 8;                   // block rows
    static constexpr int R = NB / NW;                  // block rows of a warp
    static constexpr int NBLK = NW * R * (R + 1) / 2;  // blocks a warp keeps (some of the last NW columns unused)
    __host__ __device__ static constexpr int off(int r) { return NW * r * (r + 1) / 2; }
    __host__ __device__ static constexpr int cols(int r) { return NW * (r + 1); }
    __host__ __device__ static constexpr int row(int r, int w) { return r & 1 ? r * NW + NW - 1 - w : r * NW + w; }
    __host__ __device__ static constexpr int owner(int p) { return (p / NW) & 1 ? NW - 1 - p % NW : p % NW; }
    static_assert(NB % NW == 0, "block rows per warp");
};

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
    double y[D / 8][64];            // the current panel below the pivot block, times the inverse pivots
    double w[D / 8][64];            // inverses of the unit lower triangular pivot blocks
    double dinv[D];
    double b[NRHS][D];              // right-hand sides; forward-substituted in place
    double x[NW][NRHS][D];          // solution (every warp writes its own copy)
    double part[2][NW][NRHS][8];
};

template <int NW>
__device__ __forceinline__ void sync(int bar_id) {
    if constexpr (NW == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "n"(32 * NW) : "memory");
}

// Solve for the right-hand sides in sm.b.  c: this warp's blocks of the matrix (destroyed); nba: block rows in use
// (the rest of the matrix is not touched); w, lane: warp inside the team and lane.  The solution is in sm.x[w].
// Returns false if a pivot was not positive (the same in every warp).
template <int D, int NW, int NRHS>
__device__ __forceinline__ bool solve(double (&c)[Cfg<D, NW>::NBLK][2], Smem<D, NW, NRHS>& sm, int nba, int w, int lane, int bar_id) {
    using C = Cfg<D, NW>;
    constexpr int NB = C::NB, R = C::R;
    constexpr unsigned FULL = 0xffffffffu;
    const int n = lane >> 2, t4 = lane & 3;
    double xr[R][2];
    // Pivot block p (by the warp that owns block row p): Gauss elimination on [block | I], both in accumulator layout.
    // The chain of eight steps -- shuffle, reciprocal, multiply, subtract -- is what the factorisation waits for.
    auto pivot = [&](int p, double a0, double a1) {
        double w0 = n == 2 * t4 ? 1.0 : 0.0, w1 = n == 2 * t4 + 1 ? 1.0 : 0.0, d0 = 0.0, d1 = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double col = k & 1 ? a1 : a0;
            const double piv = __shfl_sync(FULL, col, 4 * k + (k >> 1));
            const double f = __shfl_sync(FULL, col, (lane & 28) + (k >> 1));
            const double pr0 = __shfl_sync(FULL, a0, 4 * k + t4), pr1 = __shfl_sync(FULL, a1, 4 * k + t4);
            const double wr0 = __shfl_sync(FULL, w0, 4 * k + t4), wr1 = __shfl_sync(FULL, w1, 4 * k + t4);
            const double inv = fast_rcp1(piv);
            const double m = n > k ? f * inv : 0.0;
            a0 -= m * pr0;
            a1 -= m * pr1;
            w0 -= m * wr0;
            w1 -= m * wr1;
            if (2 * t4 == k) d0 = inv;
            if (2 * t4 + 1 == k) d1 = inv;
        }
        *reinterpret_cast<double2*>(&sm.w[p][2 * lane]) = make_double2(w0, w1);
        if (n == 0) *reinterpret_cast<double2*>(&sm.dinv[8 * p + 2 * t4]) = make_double2(d0, d1);
#pragma unroll
        for (int q = 0; q < NRHS; ++q) {
            double y = w0 * sm.b[q][8 * p + 2 * t4] + w1 * sm.b[q][8 * p + 2 * t4 + 1];
            y += __shfl_xor_sync(FULL, y, 1);
            y += __shfl_xor_sync(FULL, y, 2);
            __syncwarp();      // the reads of sm.b above come before the write below
            if (t4 == 0) sm.b[q][8 * p + n] = y;
        }
    };
    if (w == C::owner(0)) pivot(0, c[0][0], c[0][1]);
#pragma unroll
    for (int p = 0; p < NB; ++p) {
        if (p < nba) {
            sync<NW>(bar_id);
            const double2 wp = *reinterpret_cast<const double2*>(&sm.w[p][2 * lane]);
            const double2 di = *reinterpret_cast<const double2*>(&sm.dinv[8 * p + 2 * t4]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = C::row(r, w);
                if (C::cols(r) > p && i > p && i < nba) {
                    double* cp = c[C::off(r) + p];
                    double x0 = 0.0, x1 = 0.0;
                    dmma(x0, x1, cp[0], wp.x);
                    dmma(x0, x1, cp[1], wp.y);
                    xr[r][0] = -x0;
                    xr[r][1] = -x1;
                    cp[0] = x0 * di.x;
                    cp[1] = x1 * di.y;
                    *reinterpret_cast<double2*>(&sm.y[i][2 * lane]) = make_double2(cp[0], cp[1]);
#pragma unroll
                    for (int q = 0; q < NRHS; ++q) {
                        double s = cp[0] * sm.b[q][8 * p + 2 * t4] + cp[1] * sm.b[q][8 * p + 2 * t4 + 1];
                        s += __shfl_xor_sync(FULL, s, 1);
                        s += __shfl_xor_sync(FULL, s, 2);
                        if (t4 == 0) sm.b[q][8 * i + n] -= s;
                    }
                }
            }
            if (p + 1 < NB && p + 1 < nba) {
                sync<NW>(bar_id);
                // the next pivot block first, so that its factorisation runs beside the other warps' updates
                const int r1 = (p + 1) / NW;
                if (w == C::owner(p + 1)) {
                    const double2 yj = *reinterpret_cast<const double2*>(&sm.y[p + 1][2 * lane]);
                    double* cp = c[C::off(r1) + p + 1];
                    dmma(cp[0], cp[1], xr[r1][0], yj.x);
                    dmma(cp[0], cp[1], xr[r1][1], yj.y);
                    pivot(p + 1, cp[0], cp[1]);
                }
#pragma unroll
                for (int j = p + 1; j < NB; ++j) {
                    if (j < nba) {
                        const double2 yj = *reinterpret_cast<const double2*>(&sm.y[j][2 * lane]);
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            const int i = C::row(r, w);
                            if (C::cols(r) > j && i >= j && i > p + 1 && i < nba) {
                                double* cp = c[C::off(r) + j];
                                dmma(cp[0], cp[1], xr[r][0], yj.x);
                                dmma(cp[0], cp[1], xr[r][1], yj.y);
                            }
                        }
                    }
                }
            }
        }
    }
    sync<NW>(bar_id);
    bool ok = true;
    for (int e = lane; e < 8 * nba; e += 32)
        if (!(sm.dinv[e] > 0.0)) ok = false;
    ok = __all_sync(FULL, ok);
    // back substitution: x_p = W_p^T (D_p^{-1} y_p - sum_{i > p} Y_ip^T x_i)
#pragma unroll
    for (int p = NB - 1; p >= 0; --p) {
        if (p < nba) {
            double s[NRHS][2];
#pragma unroll
            for (int q = 0; q < NRHS; ++q) s[q][0] = s[q][1] = 0.0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = C::row(r, w);
                if (C::cols(r) > p && i > p && i < nba) {
                    const double* cp = c[C::off(r) + p];
#pragma unroll
                    for (int q = 0; q < NRHS; ++q) {
                        const double xi = sm.x[w][q][8 * i + n];
                        s[q][0] += cp[0] * xi;
                        s[q][1] += cp[1] * xi;
                    }
                }
            }
            const double2 wp = *reinterpret_cast<const double2*>(&sm.w[p][2 * lane]);
            const double dn = sm.dinv[8 * p + n];
#pragma unroll
            for (int q = 0; q < NRHS; ++q) {
#pragma unroll
                for (int o = 4; o <= 16; o <<= 1) {
                    s[q][0] += __shfl_xor_sync(FULL, s[q][0], o);
                    s[q][1] += __shfl_xor_sync(FULL, s[q][1], o);
                }
                if (lane < 4) *reinterpret_cast<double2*>(&sm.part[p & 1][w][q][2 * lane]) = make_double2(s[q][0], s[q][1]);
            }
            sync<NW>(bar_id);
#pragma unroll
            for (int q = 0; q < NRHS; ++q) {
                double v = sm.b[q][8 * p + n] * dn;
#pragma unroll
                for (int u = 0; u < NW; ++u) v -= sm.part[p & 1][u][q][n];
                double t0 = wp.x * v, t1 = wp.y * v;
#pragma unroll
                for (int o = 4; o <= 16; o <<= 1) {
                    t0 += __shfl_xor_sync(FULL, t0, o);
                    t1 += __shfl_xor_sync(FULL, t1, o);
                }
                if (lane < 4) *reinterpret_cast<double2*>(&sm.x[w][q][8 * p + 2 * lane]) = make_double2(t0, t1);
            }
            __syncwarp();
        }
    }
    return ok;
}

}  // namespace team
}  // namespace lla

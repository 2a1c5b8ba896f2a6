// Rows solved directly: explicit moments and a factorisation in fp64, on the double-precision matrix instruction.
//
// Two kinds of rows come here:
//   * rows that see fewer than head_rows keys (default 1.5 d for bf16 inputs, 2 d for fp32).  Their systems have condition
//     numbers of 1e4 .. 1e5 at the paper's ridge sizes (rank-deficient plus ridge while L < d), which the conjugate
//     gradients of the other kernels cannot resolve;
//   * every row of a problem that the tensor-core kernel does not take (fp32 inputs, d = 16) under the default solver
//     settings.  Matrix-free conjugate gradients in fp32 need 20 .. 40 sweeps of 6 d operations per (query, key) pair
//     there, explicit moments d^2 + 8 d once.
//
// A row with more than d visible keys solves the centred system C y = kbar - q of Eq. "lla_decomp",
//     C = sum_j p_j k_j k_j^T - kbar kbar^T + (lambda' / omega) I,     p_j = w_j / omega,   lambda' = lambda e^{-m},
// and o = sum_j p_j (1 - (k_j - kbar) . y) v_j.  A row with at most d keys (and a positive ridge) goes through the
// dual (Gram) form: with Z the L x d matrix of k_j - q, w_j (1 - z_j . rho) = lambda' alpha_j where
// (Z Z^T + lambda' diag(1 / w)) alpha = 1 -- a smaller system, free of the cancellation in 1 - z . rho.
//
// A block takes a few consecutive rows of a head (4 at d = 64), one team of warps each, and streams the keys through
// shared memory as doubles, a chunk at a time.  Every product is an 8 x 8 x 4 matrix instruction: scores (the block's
// query rows against eight keys), the moments (A operand w_j k_j, B operand k_j; the lower block triangle in the
// team's registers, where the factorisation continues in place: lla_team_solve.cuh), and in a second sweep k_j . y and
// the output sum (coefficients against values).  The second sweep forms the weights again instead of keeping them.
//
// What bounds it: the matrix pipe in the moments of long rows (36 of the about 47 instructions per 4 keys and row at
// d = 64; measured at 89 % of its rate), the chain of reciprocals in the pivot blocks for short ones, which the eight
// systems of two blocks on an SM hide in part.
#include "lla_team_solve.cuh"

namespace lla {
namespace {

template <int D>
struct DrCfg {
    static constexpr int NW = D == 16 ? 1 : D == 64 ? 2 : 8;      // warps per row: what the registers of 16 warps hold
    static constexpr int TEAMS = D == 128 ? 2 : 4;                // rows per block; d = 64: two blocks per SM, so that the pivot
                                                                  // chains of one run beside the products of the other
    static constexpr int WARPS = NW * TEAMS, THREADS = 32 * WARPS;
    // keys per chunk: the keys of a block with a dual row (at most d + TEAMS - 1, with a window d + TEAMS) are one chunk
    static constexpr int CH = D == 128 ? 136 : D == 64 ? 72 : 64;
    static constexpr int LDK = D + 4;                             // row stride in doubles: 4 mod 16, both operand accesses conflict-free
    static constexpr int NB = D / 8;
    static constexpr int HALVES = WARPS / NB;                     // output sum: a warp per 8 columns and part of the keys
    static constexpr int LDW = CH + 4;
};

template <int D>
struct DrSmem {
    using C = DrCfg<D>;
    double kv[C::CH][C::LDK];                 // the current chunk of keys (or values)
    double q[C::TEAMS][C::LDK];               // query rows, zero beyond the head's
    double y[C::TEAMS][C::LDK];                    // their solutions (second sweep)
    double s[C::TEAMS][C::LDW];               // scores -> weights -> output coefficients of the chunk
    double t[C::TEAMS][C::LDW];               // k_j . y
    double kbar[C::TEAMS][D];
    double gram[D <= 64 ? C::NB * (C::NB + 1) / 2 : 1][64];     // K K^T of the first d keys, 8 x 8 blocks in accumulator layout
    double osum[C::HALVES > 1 ? C::TEAMS : 1][D];   // second half of the output sum
    double red[2][C::TEAMS][C::NW];
    double den[C::TEAMS];
    team::Smem<D, C::NW, 1> solve[C::TEAMS];
};

template <typename TIn>
__device__ __forceinline__ void load_pair(const TIn* p, double& a, double& b);
template <>
__device__ __forceinline__ void load_pair<__nv_bfloat16>(const __nv_bfloat16* p, double& a, double& b) {
    const uint32_t raw = *reinterpret_cast<const uint32_t*>(p);
    a = (double)__uint_as_float(raw << 16);
    b = (double)__uint_as_float(raw & 0xFFFF0000u);
}
template <>
__device__ __forceinline__ void load_pair<float>(const float* p, double& a, double& b) {
    const float2 f = *reinterpret_cast<const float2*>(p);
    a = (double)f.x;
    b = (double)f.y;
}

// keys (or values) j0 .. j0 + CH - 1 -> shared memory; rows from jend on are zero
template <int D, typename TIn>
__device__ __forceinline__ void stage(double (*dst)[DrCfg<D>::LDK], const TIn* __restrict__ src, long long stride, int j0, int jend) {
    using C = DrCfg<D>;
    constexpr int PER = C::CH * D / 2 / C::THREADS;
    static_assert(PER * 2 * C::THREADS == C::CH * D, "a chunk is a whole number of rounds");
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int e = threadIdx.x + C::THREADS * u, j = e / (D / 2), c = 2 * (e % (D / 2));
        double a = 0.0, b = 0.0;
        if (j0 + j < jend) load_pair(src + (size_t)(j0 + j) * stride + c, a, b);
        *reinterpret_cast<double2*>(&dst[j][c]) = make_double2(a, b);
    }
}

// out[TEAMS][CH] = rows . keys, eight keys per step of a warp
template <int D>
__device__ __forceinline__ void dots(double (*out)[DrCfg<D>::LDW], const double (*rows)[DrCfg<D>::LDK], const double (*keys)[DrCfg<D>::LDK],
                                     int nkeys, int warp, int lane) {
    using C = DrCfg<D>;
    const int n = lane >> 2, t4 = lane & 3;
    for (int kb = warp; 8 * kb < nkeys; kb += C::WARPS) {
        double c[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
        for (int s = 0; s < D / 4; ++s)
            team::dmma(c[s & 1][0], c[s & 1][1], n < C::TEAMS ? rows[n][4 * s + t4] : 0.0, keys[8 * kb + n][4 * s + t4]);
        if (n < C::TEAMS) *reinterpret_cast<double2*>(&out[n][8 * kb + 2 * t4]) = make_double2(c[0][0] + c[1][0], c[0][1] + c[1][1]);
    }
}

template <int D, typename TIn, typename TOut>
__global__ void __launch_bounds__(DrCfg<D>::THREADS, D == 64 ? 2 : 1)
direct_rows_kernel(const TIn* __restrict__ q, const TIn* __restrict__ k, const TIn* __restrict__ v, TOut* __restrict__ out,
                   int n, int nq, int rows_per_head, int head_rows, int causal, double scale, double lambda, const float* __restrict__ lambda_rows,
                   int ridge_mode, float* __restrict__ rho_out, float* __restrict__ stats, int* __restrict__ iters,
                   int* __restrict__ status, int H, int kv_group, int window, const Strides sq, const Strides sk, const Strides sv,
                   const Strides so) {
    using C = DrCfg<D>;
    using T = team::Cfg<D, C::NW>;
    constexpr int NW = C::NW, TEAMS = C::TEAMS, CH = C::CH, NB = C::NB, R = T::R;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char dr_smem[];
    DrSmem<D>& sm = *reinterpret_cast<DrSmem<D>*>(dr_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const int tm = warp / NW, w = warp % NW, tt = tid % (32 * NW);      // team, warp and thread inside the team
    const int bar_id = 1 + tm;
    const int bh = blockIdx.x;                                          // heads fastest
    const int i0 = (gridDim.y - 1 - blockIdx.y) * TEAMS;                // rows with the most keys first
    const int i = i0 + tm;
    const bool live = i < rows_per_head;
    const int off = n - nq;
    const int L = !live ? 0 : causal ? off + i + 1 : n;                 // the row sees keys jlo .. L - 1
    const int jlo = causal && window > 0 ? max(0, L - window) : 0;
    const int last = min(i0 + TEAMS, rows_per_head) - 1;
    const int jend = causal ? off + last + 1 : n;                       // keys of the block
    const int jbeg = causal && window > 0 ? max(0, off + i0 + 1 - window) : 0;
    const size_t row = (size_t)bh * nq + i;
    const int hk = (bh % H) / max(kv_group, 1);
    const TIn* kb = k + sk.at(bh / H, hk, 0);
    const TIn* vb = v + sv.at(bh / H, hk, 0);

    for (int e = tid; e < TEAMS * D; e += C::THREADS) {
        const int r = e / D, c = e % D;
        sm.q[r][c] = i0 + r < rows_per_head ? (double)to_f32(q[sq.at(bh / H, bh % H, i0 + r) + c]) : 0.0;
        sm.y[r][c] = 0.0;
    }
    // one value per thread of the team -> its maximum or sum over the team
    auto team_reduce = [&](double x, bool is_max, int slot) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double z = __shfl_xor_sync(FULL, x, o);
            x = is_max ? fmax(x, z) : x + z;
        }
        if (NW > 1) {
            if (lane == 0) sm.red[slot][tm][w] = x;
            team::sync<NW>(bar_id);
            x = sm.red[slot][tm][0];
#pragma unroll
            for (int u = 1; u < NW; ++u) x = is_max ? fmax(x, sm.red[slot][tm][u]) : x + sm.red[slot][tm][u];
        }
        return x;
    };
    const double lam_i = lambda_rows && live ? (double)lambda_rows[row] : lambda;
    double c[T::NBLK][2], asum[R];
#pragma unroll
    for (int e = 0; e < T::NBLK; ++e) c[e][0] = c[e][1] = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) asum[r] = 0.0;
    // Weights are relative to m_ref, the maximum of the row's first chunk (doubles leave room for e^600 beyond it,
    // after which everything is rescaled); m_max is the true maximum, which the outputs refer to.
    double m_ref = -INFINITY, m_max = -INFINITY, omega = 0.0, lam_m = 0.0;
    // at most d keys: the dual form.  (lambda' could only vanish if lambda does.)
    const bool dual = live && L <= D && jlo == 0 && jbeg == 0 && jend <= CH && lam_i > 0.0;

    // ---- first sweep: weights and moments ----
    for (int j0 = jbeg; j0 < jend; j0 += CH) {
        const int nk = min(CH, jend - j0);
        __syncthreads();
        stage<D>(sm.kv, kb, sk.r, j0, jend);
        __syncthreads();
        dots<D>(sm.s, sm.q, sm.kv, nk, warp, lane);
        if (D <= 64 && jend <= CH && (causal ? off + i0 + 1 : n) <= D) {        // a row of the block may be dual
            for (int e = warp, bi = 0; e < NB * (NB + 1) / 2; e += C::WARPS) {
                while ((bi + 1) * (bi + 2) / 2 <= e) ++bi;
                const int bj = e - bi * (bi + 1) / 2;
                if (8 * bi >= nk) continue;
                double x[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
                for (int s = 0; s < D / 4; ++s) team::dmma(x[s & 1][0], x[s & 1][1], sm.kv[8 * bi + g][4 * s + t4], sm.kv[8 * bj + g][4 * s + t4]);
                *reinterpret_cast<double2*>(&sm.gram[e][2 * lane]) = make_double2(x[0][0] + x[1][0], x[0][1] + x[1][1]);
            }
        }
        __syncthreads();
        if (j0 >= L || j0 + CH <= jlo) continue;                          // (uniform over the team) no key of this row
        double cmax = -INFINITY;
        for (int j = tt; j < nk; j += 32 * NW) {
            const bool vis = j0 + j < L && j0 + j >= jlo;
            if (vis) cmax = fmax(cmax, sm.s[tm][j] * scale);
        }
        cmax = team_reduce(cmax, true, 0);
        m_max = fmax(m_max, cmax);
        if (m_ref == -INFINITY) {
            m_ref = cmax;
        } else if (cmax > m_ref + 600.0) {
            const double f = exp(m_ref - cmax);
#pragma unroll
            for (int e = 0; e < T::NBLK; ++e) { c[e][0] *= f; c[e][1] *= f; }
#pragma unroll
            for (int r = 0; r < R; ++r) asum[r] *= f;
            omega *= f;
            m_ref = cmax;
        }
        for (int j = tt; j < CH; j += 32 * NW) {
            const bool vis = j < nk && j0 + j < L && j0 + j >= jlo;
            const double sj = sm.s[tm][j], e = vis ? exp(sj * scale - m_ref) : 0.0;
            if (dual) sm.t[tm][j] = sj;
            sm.s[tm][j] = e;
            omega += e;
        }
        team::sync<NW>(bar_id);
        if (!dual) {
            // keys 4 s + t4: A operand w_j k_j of this warp's block rows, B operand k_j of every block column
            const int ns = (min(nk, L - j0) + 3) / 4;
            team::with_warp<NW>(w, [&](auto wc) {
                constexpr int W = decltype(wc)::value;
#pragma unroll(D == 16 ? 4 : 1)
                for (int s = 0; s < ns; ++s) {
                    const double* kr = sm.kv[4 * s + t4] + g;
                    const double wj = sm.s[tm][4 * s + t4];
                    double av[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        av[r] = wj * kr[8 * T::row(r, W)];
                        asum[r] += av[r];
                    }
#pragma unroll
                    for (int j = 0; j <= T::row(R - 1, W); ++j) {
                        const double bv = kr[8 * j];
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            if (j <= T::row(r, W)) team::dmma(c[T::off(r) + j][0], c[T::off(r) + j][1], av[r], bv);
                    }
                }
            });
        }
    }
    // team-wide sums (every team has run every block barrier above)
    if (live) {
        omega = team_reduce(omega, false, 1);
        lam_m = ridge_mode == LLA_RIDGE_PRINTED ? lam_i * exp(m_max - m_ref) : lam_i * exp(-m_ref);
    }
    const double inv = 1.0 / omega;
    team::Smem<D, NW, 1>& ss = sm.solve[tm];
    bool ok = true;
    int nba = NB;
    if (dual) {
        // The block's keys are one chunk and still in shared memory (jlo = 0: a window is never shorter than the rows
        // that see at most d keys).  Row and column index: the key; the padding to a multiple of eight is an identity block.
        // z_j . z_l = k_j . k_l - k_j . q - k_l . q + q . q; the first product is the same for the block's rows (it has
        // them in shared memory at d <= 64: 576 instead of 576 per row instructions at 64 keys).  Rows of the chunk past
        // the block's keys are zero.
        nba = (L + 7) / 8;
        if constexpr (D <= 64) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int bi = T::row(r, w);
#pragma unroll
                for (int j = 0; j < NB; ++j)
                    if (T::cols(r) > j && j <= bi && bi < nba) {
                        const double2 x = *reinterpret_cast<const double2*>(&sm.gram[bi * (bi + 1) / 2 + j][2 * lane]);
                        c[T::off(r) + j][0] = x.x;
                        c[T::off(r) + j][1] = x.y;
                    }
            }
        } else {
            team::with_warp<NW>(w, [&](auto wc) {
                constexpr int W = decltype(wc)::value;
                for (int s = 0; s < D / 4; ++s) {
                    const double* kr = sm.kv[g] + 4 * s + t4;
                    double av[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) av[r] = kr[8 * C::LDK * T::row(r, W)];
#pragma unroll
                    for (int j = 0; j <= T::row(R - 1, W); ++j) {
                        if (j >= nba) break;
                        const double bv = kr[8 * C::LDK * j];
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            if (j <= T::row(r, W)) team::dmma(c[T::off(r) + j][0], c[T::off(r) + j][1], av[r], bv);
                    }
                }
            });
        }
        double qq = 0.0;
        for (int e = lane; e < D; e += 32) qq += sm.q[tm][e] * sm.q[tm][e];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) qq += __shfl_xor_sync(FULL, qq, o);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int bi = T::row(r, w), idx = 8 * bi + g;
            const double si = qq - sm.t[tm][idx];
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (T::cols(r) > j && j <= bi && bi < nba) {
                    double* cp = c[T::off(r) + j];
                    const int jdx = 8 * j + 2 * t4;
                    const bool in0 = idx < L && jdx < L, in1 = idx < L && jdx + 1 < L;
                    cp[0] = in0 ? cp[0] + (si - sm.t[tm][jdx]) : 0.0;
                    cp[1] = in1 ? cp[1] + (si - sm.t[tm][jdx + 1]) : 0.0;
                    if (j == bi) {
                        // ridge over weight for live keys (weights kept away from zero), one for the padding
                        const double dg = idx < L ? lam_m / fmax(sm.s[tm][idx], 1e-290) : 1.0;
                        if (g == 2 * t4) cp[0] += dg;
                        if (g == 2 * t4 + 1) cp[1] += dg;
                    }
                }
        }
        for (int e = tt; e < 8 * nba; e += 32 * NW) ss.b[0][e] = e < L ? 1.0 : 0.0;
    } else if (live) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double a = asum[r];
            a += __shfl_xor_sync(FULL, a, 1);
            a += __shfl_xor_sync(FULL, a, 2);
            const int cc = 8 * T::row(r, w) + g;
            if (t4 == 0) {
                sm.kbar[tm][cc] = a * inv;
                ss.b[0][cc] = a * inv - sm.q[tm][cc];
            }
        }
        team::sync<NW>(bar_id);
        const double ridge = lam_m * inv;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int bi = T::row(r, w);
            const double kr = sm.kbar[tm][8 * bi + g];
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (T::cols(r) > j && j <= bi) {
                    double* cp = c[T::off(r) + j];
                    const double2 kc = *reinterpret_cast<const double2*>(&sm.kbar[tm][8 * j + 2 * t4]);
                    cp[0] = cp[0] * inv - kr * kc.x;
                    cp[1] = cp[1] * inv - kr * kc.y;
                    if (j == bi) {
                        if (g == 2 * t4) cp[0] += ridge;
                        if (g == 2 * t4 + 1) cp[1] += ridge;
                    }
                }
        }
    }
    double ybar = 0.0, gfac = 1.0, csum = 0.0;
    if (live) {
        team::sync<NW>(bar_id);
        if constexpr (NW <= 2) team::with_warp<NW>(w, [&](auto wc) { ok = team::solve<D, NW, 1>(c, ss, nba, decltype(wc)::value, lane, bar_id); });
        else ok = team::solve<D, NW, 1>(c, ss, nba, w, lane, bar_id);
        team::sync<NW>(bar_id);
        if (dual) {
            // coefficients lambda' alpha_j over the chunk's keys
            for (int j = tt; j < CH; j += 32 * NW) {
                const double cj = j < L ? lam_m * ss.x[w][0][j] : 0.0;
                sm.s[tm][j] = cj;
                csum += cj;
            }
            if (rho_out)                                                   // rho = Z^T alpha
                for (int e = tt; e < D; e += 32 * NW) {
                    double a = 0.0;
                    for (int j = 0; j < L; ++j) a += ss.x[w][0][j] * (sm.kv[j][e] - sm.q[tm][e]);
                    rho_out[row * D + e] = (float)a;
                }
        } else {
            double yb = 0.0, yk = 0.0;
            for (int e = lane; e < D; e += 32) {
                const double y = ss.x[w][0][e], kbv = sm.kbar[tm][e];
                yk += kbv * y;
                yb += (kbv - sm.q[tm][e]) * y;
                if (w == 0) sm.y[tm][e] = y;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                yk += __shfl_xor_sync(FULL, yk, o);
                yb += __shfl_xor_sync(FULL, yb, o);
            }
            ybar = yk;
            gfac = 1.0 + yb;
            if (rho_out && w == 0)
                for (int e = lane; e < D; e += 32) rho_out[row * D + e] = (float)(ss.x[w][0][e] / gfac);
        }
    }
    // ---- second sweep: coefficients and output ----
    const int ob = warp % NB, half = warp / NB;
    double o0 = 0.0, o1 = 0.0;
    const bool one_chunk = jend - jbeg <= CH;
    for (int j0 = jbeg; j0 < jend; j0 += CH) {
        const int nk = min(CH, jend - j0);
        __syncthreads();
        if (!one_chunk) {
            stage<D>(sm.kv, kb, sk.r, j0, jend);
            __syncthreads();
            dots<D>(sm.s, sm.q, sm.kv, nk, warp, lane);         // (a dual row's block is one chunk)
        }
        dots<D>(sm.t, sm.y, sm.kv, nk, warp, lane);
        __syncthreads();
        if (!dual)
            for (int j = tt; j < CH; j += 32 * NW) {
                const bool vis = j < nk && j0 + j < L && j0 + j >= jlo;
                double cj = 0.0;
                if (vis) {
                    const double e = one_chunk ? sm.s[tm][j] : exp(sm.s[tm][j] * scale - m_ref);
                    cj = e * (1.0 - (sm.t[tm][j] - ybar));
                }
                sm.s[tm][j] = cj;
                csum += cj;
            }
        stage<D>(sm.kv, vb, sv.r, j0, jend);
        __syncthreads();
        if (half < C::HALVES) {
            const int s1 = (nk + 3) / 4;
            for (int s = half; s < s1; s += C::HALVES)
                team::dmma(o0, o1, g < TEAMS ? sm.s[g][4 * s + t4] : 0.0, sm.kv[4 * s + t4][8 * ob + g]);
        }
    }
    const double den = team_reduce(csum, false, 0);
    if (tt == 0) sm.den[tm] = den;
    if (C::HALVES > 1 && half == 1 && g < TEAMS) *reinterpret_cast<double2*>(&sm.osum[g][8 * ob + 2 * t4]) = make_double2(o0, o1);
    __syncthreads();
    if (half == 0 && g < TEAMS && i0 + g < rows_per_head) {
        if (C::HALVES > 1) {
            const double2 p = *reinterpret_cast<const double2*>(&sm.osum[g][8 * ob + 2 * t4]);
            o0 += p.x;
            o1 += p.y;
        }
        const double id = 1.0 / sm.den[g];
        TOut* orow = out + so.at(bh / H, bh % H, i0 + g) + 8 * ob + 2 * t4;
        if (LLA_IN_BOUNDS((size_t)bh * nq + i0 + g, (size_t)gridDim.x * nq, status, 201)) {
            store_out(orow, (float)(o0 * id));
            store_out(orow + 1, (float)(o1 * id));
        }
    }
    if (live && tt == 0) {
        if (stats) {
            const double f = exp(m_ref - m_max);       // to weights relative to the true maximum
            const double om = omega * f, dl = dual ? den * f : omega * f / gfac;
            stats[row * 3 + 0] = (float)m_max;
            stats[row * 3 + 1] = (float)om;
            stats[row * 3 + 2] = (float)dl;
        }
        if (iters) iters[row] = L < head_rows ? -1 : 0;      // (0: a row that conjugate gradients could have solved)
        if (!ok && status) atomicAdd(status + LLA_STATUS_BAD_PIVOT, 1);
    }
}

template <int D, typename TIn, typename TOut>
int launch_t(const ForwardArgs& a, int rows) {
    using C = DrCfg<D>;
    static_assert(C::HALVES <= 2 && C::HALVES * C::NB == C::WARPS, "output sum layout");
    const int smem = (int)sizeof(DrSmem<D>);
    auto kern = direct_rows_kernel<D, TIn, TOut>;
    LLA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    LLA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    dim3 grid(a.B * a.H, (rows + C::TEAMS - 1) / C::TEAMS);
    kern<<<grid, C::THREADS, smem, a.stream>>>((const TIn*)a.q, (const TIn*)a.k, (const TIn*)a.v, (TOut*)a.out, a.n, a.nq, rows, a.head_rows, a.causal,
                                               (double)a.scale, (double)a.lambda, a.lambda_rows, a.ridge_mode, a.rho, a.stats, a.iters,
                                               a.status, a.H, a.kv_group, a.window, a.sq, a.sk, a.sv, a.so);
    LLA_CUDA_TRY(cudaGetLastError());
    return LLA_OK;
}

template <int D>
int launch_d(const ForwardArgs& a, int rows) {
    if (a.in_dtype == LLA_BF16 && a.out_dtype == LLA_BF16) return launch_t<D, __nv_bfloat16, __nv_bfloat16>(a, rows);
    if (a.in_dtype == LLA_BF16 && a.out_dtype == LLA_F32) return launch_t<D, __nv_bfloat16, float>(a, rows);
    if (a.in_dtype == LLA_F32 && a.out_dtype == LLA_F32) return launch_t<D, float, float>(a, rows);
    return LLA_ERR_UNSUPPORTED;
}

}  // namespace

// Number of leading rows per head handled directly (causal), or nq / 0 (non-causal).
int head_rows_count(const ForwardArgs& a) {
    if (a.all_direct) return a.nq;
    if (a.head_rows <= 0) return 0;
    if (a.causal) {     // query row i sees n - nq + i + 1 keys
        const int rows = a.head_rows - 1 - (a.n - a.nq);
        return rows < 0 ? 0 : (rows > a.nq ? a.nq : rows);
    }
    return a.n < a.head_rows ? a.nq : 0;
}

int launch_head_rows(const ForwardArgs& a) {
    const int rows = head_rows_count(a);
    if (rows <= 0) return LLA_OK;
    if (a.d != a.dv) return LLA_ERR_UNSUPPORTED;
    switch (a.d) {
        case 16: return launch_d<16>(a, rows);
        case 64: return launch_d<64>(a, rows);
        case 128: return launch_d<128>(a, rows);
        default: return LLA_ERR_UNSUPPORTED;
    }
}

}  // namespace lla

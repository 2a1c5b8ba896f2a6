// Rows solved directly: explicit moments and a factorisation in fp64, on the double-precision matrix instruction.
//
// Two kinds of rows come here:
//   * rows that see fewer than head_rows keys (default 1.5 d for bf16 inputs, 2 d for fp32).  Their systems have condition
//     numbers of 1e4 .. 1e5 at the paper's ridge sizes (rank-deficient plus ridge while L < d), which the conjugate
//     gradients of the other kernels cannot resolve;
//   * the rows of a problem that the tensor-core kernel does not take (fp32 inputs, d = 16) under the default solver
//     settings, all of them or up to a number of keys (direct_rows_worthwhile below).  Matrix-free conjugate gradients
//     in fp32 need 10 .. 40 sweeps of 6 d operations per (query, key) pair there, explicit moments d^2 + 8 d once.
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
// team's registers, then in shared memory over the keys for the factorisation: lla_team_solve.cuh), and in a second
// sweep k_j . y and the output sum (coefficients against values).  The second sweep forms the weights again instead of keeping them.
//
// fp32 inputs may lie far from the origin compared with their spread, up to 2^24 times, and squares of that do not fit a
// double's 53 bits beside the spread's and a small ridge.  So in the blocks with ill-conditioned rows (fewer than head_rows
// keys) their keys are staged relative to the block's first query, the ridge corrected by its product with the row's
// query; and where the rounding of the shared products is not far below the ridge, the dual form's matrix is
// formed from the differences k_j - q themselves, row by row.  (bf16 inputs reach 2^8 at most: products of the keys as they
// are lose nothing.)  Both measured at 8 fp32 heads, d = 64: n = 1000, keys of every block shifted 1069 us, of those blocks
// 1023 us; n = 63, all matrices row by row 39 us, shared 33 us.
//
// What bounds it: the matrix pipe in the moments of long rows (36 of the about 47 instructions per 4 keys and row at
// d = 64; measured at 89 % of its rate), the chain of reciprocals in the pivot blocks for short ones, which the eight
// systems of two blocks on an SM hide in part.
#include <algorithm>

#include "lla_rows.cuh"

namespace lla {
namespace {

template <int D, bool REL>
struct DrSmem {
    using C = DrCfg<D>;
    union {
        double kv[C::CH][C::LDK];                                  // the current chunk of keys (or values)
        double mat[C::TEAMS][team::Cfg<D, C::NW>::LOWER][64];      // the systems, between the sweeps
    };
    double q[C::TEAMS][C::LDK];               // query rows, zero beyond the head's
    double rel[REL ? C::TEAMS + 1 : 1][C::LDK];    // REL: the same minus the first of them; the first (zero where it is not finite)
    double y[C::TEAMS][C::LDK];                    // their solutions (second sweep)
    double s[C::TEAMS][C::LDW];               // scores -> weights -> output coefficients of the chunk
    double t[C::TEAMS][C::LDW];               // k_j . y
    double kbar[C::TEAMS][D];
    double osum[C::HALVES > 1 ? C::TEAMS : 1][D];   // second half of the output sum
    double red[2][C::TEAMS][C::NW];
    double den[C::TEAMS], lam[C::TEAMS], qq[C::TEAMS], qn[REL ? C::TEAMS : 1];      // qq: |q|^2 in the frame of the keys; qn: |q|^2
    double kmax[REL ? C::WARPS : 1];
    int dual[C::TEAMS];                       // visible keys of a dual row, 0 for the others
    unsigned bad[2];                          // keys, values at the ends of the block's range that are not finite (see Ends)
    team::Smem<D, C::NW, 1> solve[C::TEAMS];
};

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
    constexpr bool REL = sizeof(TIn) == 4;             // keys relative to the block's first query
    extern __shared__ __align__(16) unsigned char dr_smem[];
    DrSmem<D, REL>& sm = *reinterpret_cast<DrSmem<D, REL>*>(dr_smem);
    auto row_of = [](auto& rows) { return [&rows](int r) { return &rows[r][0]; }; };
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
    const int ch = jend - jbeg <= CH ? CH : C::STEP;                    // keys per chunk
    const size_t row = (size_t)bh * nq + i;
    const int hk = (bh % H) / max(kv_group, 1);
    const TIn* kb = k + sk.at(bh / H, hk, 0);
    const TIn* vb = v + sv.at(bh / H, hk, 0);

    for (int e = tid; e < TEAMS * D; e += C::THREADS) {
        const int r = e / D, c = e % D;
        sm.q[r][c] = i0 + r < rows_per_head ? (double)to_f32(q[sq.at(bh / H, bh % H, i0 + r) + c]) : 0.0;
        sm.y[r][c] = 0.0;
    }
    const bool rel = REL && (causal ? off + i0 + 1 : n) < head_rows;
    const double* qc = rel ? sm.rel[tm] : sm.q[tm];                     // the row's query in the frame of the staged keys
    if (rel) {
        __syncthreads();
        for (int e = tid; e < (TEAMS + 1) * D; e += C::THREADS) {
            const int r = e / D, c = e % D;
            const double x = sm.q[0][c], ref = isfinite(x) ? x : 0.0;
            sm.rel[r][c] = r < TEAMS ? sm.q[r][c] - ref : ref;
        }
    }
    if (tid < 2) sm.bad[tid] = 0u;
    auto ends = [&]() {
        const int e = off + i0 + 1;
        return Ends{causal ? e : 0, causal ? off + last + 1 : 0, jbeg, causal && window > 0 ? max(0, off + last + 1 - window) : 0};
    };
    auto checked = [&](int j0, int nk, int what) {                      // the chunk's ends, before the barrier that ends its staging
        if (causal) take_out<D>(sm.kv, off + i0 + 1 - j0, nk, 1u, &sm.bad[what]);
        if (causal && window > 0) take_out<D>(sm.kv, jbeg - j0, nk, 256u, &sm.bad[what]);
    };
    auto stage_keys = [&](int j0) {
        if (rel) stage<D, true>(sm.kv, kb, sk.r, j0, jend, ch, sm.rel[TEAMS]);
        else stage<D>(sm.kv, kb, sk.r, j0, jend, ch);
    };
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
    for (int j0 = jbeg; j0 < jend; j0 += ch) {
        const int nk = min(ch, jend - j0);
        __syncthreads();
        stage_keys(j0);
        checked(j0, nk, 0);
        __syncthreads();
        dots<D>(row_of(sm.s), row_of(sm.q), sm.kv, nk, warp, lane);
        __syncthreads();
        if (j0 >= L || j0 + ch <= jlo) continue;                          // (uniform over the team) no key of this row
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
        for (int j = tt; j < ch; j += 32 * NW) {
            const bool vis = j < nk && j0 + j < L && j0 + j >= jlo;
            const double sj = sm.s[tm][j], e = vis ? exp(sj * scale - m_ref) : 0.0;
            sm.t[tm][j] = sj;                          // (kept for the dual form)
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
    // What the frame of the keys takes from the row's scores.  (The weights are relative to the maximum and need it nowhere.)
    auto frame = [&]() {
        double x = 0.0;
        if (rel) {
            for (int e = lane; e < D; e += 32) x += sm.q[tm][e] * sm.rel[TEAMS][e];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
        }
        return x * scale;
    };
    // team-wide sums (every team has run every block barrier above)
    if (live) {
        omega = team_reduce(omega, false, 1);
        lam_m = ridge_mode == LLA_RIDGE_PRINTED ? lam_i : lam_i * exp(-(m_max + frame()));      // beside weights relative to m_max
    }
    const double inv = 1.0 / omega;
    team::Smem<D, NW, 1>& ss = sm.solve[tm];
    bool ok = true;
    const int nba = dual ? (L + 7) / 8 : NB;
    sm.dual[tm] = dual ? L : 0;
    sm.lam[tm] = lam_m;
    if (dual) {
        // the diagonal of the dual form: ridge over weight for live keys (weights kept away from zero); the padding to a
        // multiple of eight is an identity block
        for (int j = tt; j < 8 * nba; j += 32 * NW) sm.s[tm][j] = j < L ? lam_m / fmax(sm.s[tm][j], 1e-290) : 1.0;
    }
    if (dual && w == 0) {
        double qq = 0.0, qn = 0.0;
        for (int e = lane; e < D; e += 32) {
            qq += qc[e] * qc[e];
            if (REL) qn += sm.q[tm][e] * sm.q[tm][e];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            qq += __shfl_xor_sync(FULL, qq, o);
            if (REL) qn += __shfl_xor_sync(FULL, qn, o);
        }
        if (lane == 0) {
            sm.qq[tm] = qq;
            if (REL) sm.qn[tm] = qn;
        }
    }
    if (live && !dual) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double a = asum[r];
            a += __shfl_xor_sync(FULL, a, 1);
            a += __shfl_xor_sync(FULL, a, 2);
            const int cc = 8 * T::row(r, w) + g;
            if (t4 == 0) {
                sm.kbar[tm][cc] = a * inv;
                ss.b[0][cc] = a * inv - qc[cc];
            }
        }
    }
    // Dual rows of the block (its first keys are one chunk, still in shared memory; jlo = 0, for a window is never
    // shorter than the rows that see at most d keys): z_j . z_l = k_j . k_l - k_j . q - k_l . q + q . q, of which the
    // first product is the same for all of them.  The block's warps share its blocks out, and each
    // writes a block of K K^T, corrected, into every dual row's matrix.
    constexpr int GB = (T::LOWER + C::WARPS - 1) / C::WARPS;
    double gm[GB][2];
    const bool some_dual = jbeg == 0 && jend <= CH && (causal ? off + i0 + 1 : n) <= D;
    bool rowwise = false;
    if (some_dual) {
        double kmax = 0.0;
#pragma unroll
        for (int u = 0; u < GB; ++u) {
            const int e = warp + C::WARPS * u;
            int bi = 0;
            while ((bi + 1) * (bi + 2) / 2 <= e) ++bi;
            const int bj = e - team::blk(bi, 0);
            gm[u][0] = gm[u][1] = 0.0;
            if (e < T::LOWER && 8 * bi < jend) {
                double x[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 8
                for (int s = 0; s < D / 4; ++s) team::dmma(x[s & 1][0], x[s & 1][1], sm.kv[8 * bi + g][4 * s + t4], sm.kv[8 * bj + g][4 * s + t4]);
                gm[u][0] = x[0][0] + x[1][0];
                gm[u][1] = x[0][1] + x[1][1];
                if (REL && bi == bj && 8 * bi + g < jend) kmax = fmax(kmax, g == 2 * t4 ? gm[u][0] : g == 2 * t4 + 1 ? gm[u][1] : 0.0);
            }
        }
        if (REL) {
            // the rounding of the products below, 1e-16 of the largest |k|^2 or |k| |q|, against the ridge
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) kmax = fmax(kmax, __shfl_xor_sync(FULL, kmax, o));
            if (lane == 0) sm.kmax[warp] = kmax;
            __syncthreads();
#pragma unroll
            for (int u = 0; u < C::WARPS; ++u) kmax = fmax(kmax, sm.kmax[u]);
            rowwise = !isfinite(sm.qn[0]);                 // (the products below take that query's from the others')
            for (int t = 0; t < TEAMS; ++t)
                rowwise = rowwise || (sm.dual[t] && !(sm.lam[t] >= 1e-8 * fmax(fmax(kmax, sm.qq[t]), sqrt(kmax * sm.qn[t]))));
        }
    }
    // a dual row's matrix from its own differences, in the place of the moments
    if (REL && rowwise && dual) {
        team::with_warp<NW>(w, [&](auto wc) {
            constexpr int W = decltype(wc)::value;
#pragma unroll 1
            for (int s = 0; s < D / 4; ++s) {
                const double qe = qc[4 * s + t4];
                auto z = [&](int b) { return 8 * b + g < L ? sm.kv[8 * b + g][4 * s + t4] - qe : 0.0; };
                double av[R];
#pragma unroll
                for (int r = 0; r < R; ++r) av[r] = z(T::row(r, W));
#pragma unroll
                for (int j = 0; j <= T::row(R - 1, W); ++j) {
                    if (j >= nba) break;
                    const double bv = z(j);
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (j <= T::row(r, W)) team::dmma(c[T::off(r) + j][0], c[T::off(r) + j][1], av[r], bv);
                }
            }
        });
    }
    __syncthreads();               // the keys are no longer read: their place takes the matrices
    if (some_dual && !rowwise) {
#pragma unroll
        for (int u = 0; u < GB; ++u) {
            const int e = warp + C::WARPS * u;
            if (e >= T::LOWER) break;
            int bi = 0;
            while ((bi + 1) * (bi + 2) / 2 <= e) ++bi;
            const int bj = e - team::blk(bi, 0), idx = 8 * bi + g, jdx = 8 * bj + 2 * t4;
            for (int t = 0; t < TEAMS; ++t) {
                const int Lt = sm.dual[t];
                if (8 * bi >= Lt) continue;
                // q . k_j (REL: k_j relative to the block's first query, whose product goes off)
                auto qk = [&](int j) { return REL ? sm.t[t][j] - sm.t[0][j] : sm.t[t][j]; };
                const double si = sm.qq[t] - (idx < Lt ? qk(idx) : 0.0);
                double v0 = idx < Lt && jdx < Lt ? gm[u][0] + (si - qk(jdx)) : 0.0;
                double v1 = idx < Lt && jdx + 1 < Lt ? gm[u][1] + (si - qk(jdx + 1)) : 0.0;
                if (bi == bj) {
                    const double dg = sm.s[t][idx];
                    if (g == 2 * t4) v0 += dg;
                    if (g == 2 * t4 + 1) v1 += dg;
                }
                *reinterpret_cast<double2*>(&sm.mat[t][e][2 * lane]) = make_double2(v0, v1);
            }
        }
    }
    if (dual) {
        for (int e = tt; e < 8 * nba; e += 32 * NW) ss.b[0][e] = e < L ? 1.0 : 0.0;
        if (REL && rowwise) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int bi = T::row(r, w);
                if (bi >= nba) continue;
                const double dg = sm.s[tm][8 * bi + g];
#pragma unroll
                for (int j = 0; j < NB; ++j)
                    if (T::cols(r) > j && j <= bi) {
                        double v0 = c[T::off(r) + j][0], v1 = c[T::off(r) + j][1];
                        if (j == bi) {
                            if (g == 2 * t4) v0 += dg;
                            if (g == 2 * t4 + 1) v1 += dg;
                        }
                        *reinterpret_cast<double2*>(&sm.mat[tm][team::blk(bi, j)][2 * lane]) = make_double2(v0, v1);
                    }
            }
        }
    } else if (live) {
        const double ridge = lam_m * (inv * exp(m_max - m_ref));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int bi = T::row(r, w);
            const double kr = sm.kbar[tm][8 * bi + g];
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (T::cols(r) > j && j <= bi) {
                    const double2 kc = *reinterpret_cast<const double2*>(&sm.kbar[tm][8 * j + 2 * t4]);
                    double v0 = c[T::off(r) + j][0] * inv - kr * kc.x, v1 = c[T::off(r) + j][1] * inv - kr * kc.y;
                    if (j == bi) {
                        if (g == 2 * t4) v0 += ridge;
                        if (g == 2 * t4 + 1) v1 += ridge;
                    }
                    *reinterpret_cast<double2*>(&sm.mat[tm][team::blk(bi, j)][2 * lane]) = make_double2(v0, v1);
                }
        }
    }
    if (some_dual) __syncthreads();
    double ybar = 0.0, gfac = 1.0, csum = 0.0;
    if (live) {
        team::sync<NW>(bar_id);
        ok = team::solve<D, NW, 1>(sm.mat[tm], ss, nba, w, lane, bar_id);
        if (dual) {
            // coefficients lambda' alpha_j over the chunk's keys
            for (int j = tt; j < CH; j += 32 * NW) {
                const double cj = j < L ? lam_m * ss.x[w][0][j] : 0.0;
                sm.s[tm][j] = cj;
                csum += cj;
            }
        } else {
            double yb = 0.0, yk = 0.0;
            for (int e = lane; e < D; e += 32) {
                const double y = ss.x[w][0][e], kbv = sm.kbar[tm][e];
                yk += kbv * y;
                yb += (kbv - qc[e]) * y;
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
    // (a block of dual rows needs its keys again only for rho)
    const bool keys = !some_dual || rho_out || (causal ? off + last + 1 : n) > D || lambda_rows || lambda == 0.0;
    for (int j0 = jbeg; j0 < jend; j0 += ch) {
        const int nk = min(ch, jend - j0);
        __syncthreads();
        if (keys) {
            stage_keys(j0);
            checked(j0, nk, 0);
            __syncthreads();
            if (dual) {
                if (rho_out)                                       // rho = Z^T alpha
                    for (int e = tt; e < D; e += 32 * NW) {
                        double a = 0.0;
                        for (int j = 0; j < L; ++j) a += ss.x[w][0][j] * (sm.kv[j][e] - qc[e]);
                        rho_out[row * D + e] = (float)a;
                    }
            }
            // scores again, except in a block of one chunk, which still has the weights
            if (jend - jbeg > CH) dots<D>(row_of(sm.s), row_of(sm.q), sm.kv, nk, warp, lane);
        }
        if (keys) dots<D>(row_of(sm.t), row_of(sm.y), sm.kv, nk, warp, lane);
        __syncthreads();
        if (!dual)
            for (int j = tt; j < ch; j += 32 * NW) {
                const bool vis = j < nk && j0 + j < L && j0 + j >= jlo;
                double cj = 0.0;
                if (vis) {
                    const double e = jend - jbeg <= CH ? sm.s[tm][j] : exp(sm.s[tm][j] * scale - m_ref);
                    cj = e * (1.0 - (sm.t[tm][j] - ybar));
                }
                sm.s[tm][j] = cj;
                csum += cj;
            }
        stage<D>(sm.kv, vb, sv.r, j0, jend, ch);
        checked(j0, nk, 1);
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
        if (sm.bad[0] | sm.bad[1]) {
            const double2 x = spoilt(sm.bad, ends(), g, causal && window > 0 ? max(0, off + i0 + g + 1 - window) : 0, vb + 8 * ob + 2 * t4, sv.r);
            o0 += x.x;
            o1 += x.y;
        }
        TOut* orow = out + so.at(bh / H, bh % H, i0 + g) + 8 * ob + 2 * t4;
        if (LLA_IN_BOUNDS((size_t)bh * nq + i0 + g, (size_t)gridDim.x * nq, status, 201)) {
            store_out(orow, (float)(o0 * id));
            store_out(orow + 1, (float)(o1 * id));
        }
    }
    const double f = exp(m_ref - m_max);           // to weights relative to the true maximum
    if (live && stats) m_max += frame();           // (by whole warps)
    bool spoil = false;                            // the row sees a key that is not finite
    if (live && sm.bad[0]) {
        spoil = (sm.bad[0] & ends().seen(tm, jlo)) != 0u;
        if (spoil && rho_out && w == 0)
            for (int e = lane; e < D; e += 32) rho_out[row * D + e] = NAN;
    }
    if (live && tt == 0) {
        if (stats) {
                        const double om = omega * f, dl = dual ? den * f : omega * f / gfac;
            stats[row * 3 + 0] = (float)m_max;
            stats[row * 3 + 1] = spoil ? NAN : (float)om;
            stats[row * 3 + 2] = spoil ? NAN : (float)dl;
        }
        if (iters) iters[row] = L < head_rows ? -1 : 0;      // (0: a row that conjugate gradients could have solved)
        if (!ok && status) atomicAdd(status + LLA_STATUS_BAD_PIVOT, 1);
    }
}

template <int D, typename TIn, typename TOut>
int launch_t(const ForwardArgs& a, int rows) {
    using C = DrCfg<D>;
    static_assert(C::HALVES <= 2 && C::HALVES * C::NB == C::WARPS, "output sum layout");
    const int smem = (int)sizeof(DrSmem<D, sizeof(TIn) == 4>);
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

constexpr int kMaxRowBlocks = 65535;      // blocks of rows in the second dimension of the grid

int direct_rows_below(const ForwardArgs& a) { return std::max(a.head_rows, a.direct_below); }

// Direct or fp32 conjugate gradients (lla_forward_simt.cu), for problems that the tensor-core kernel does not take.  A row
// with L keys costs here kd L + c0 microseconds of an SM whatever the data, there about ks L + s0 (keys and queries of the
// usual recipe; the iterations fall with L, sharper weights take more).  Measured:
//     d = 128: 0.137 L + 10    0.0575 L + 50    equal at 500 keys   (16 heads, n = 4000: 121 ms direct, 73 ms)
//     d = 64:  0.031 L + 2.5   0.0194 L + 35    equal at 2800 keys  (8 heads, n = 8000: 54 ms direct, 50 ms)
//     d = 16:  0.0067 L + 0.5  0.0056 L + 7.4   equal at 6300 keys  (16 heads, n = 8000: 23 ms direct, 26 ms)
// But conjugate gradients are as slow as their longest block, which takes its rows through all sweeps alone (2 heads, n =
// 2000, d = 128: 4.1 ms direct, 5.5 ms): the rows from that line on go there only if the whole call is shorter for it.
// (And with a window, which keeps the keys few however long the sequence, those that a launch has no blocks left for.)
int direct_rows_worthwhile(const ForwardArgs& a) {
    const double kd = a.d == 128 ? 0.137 : a.d == 64 ? 0.031 : 0.0067, c0 = a.d == 128 ? 10.0 : a.d == 64 ? 2.5 : 0.5;
    const double ks = a.d == 128 ? 0.0575 : a.d == 64 ? 0.0194 : 0.0056, s0 = a.d == 128 ? 50.0 : a.d == 64 ? 35.0 : 7.4;
    const int block_rows = a.d == 128 ? 32 : 64, off = a.n - a.nq;
    const long long room = off + kMaxRowBlocks * (a.d == 128 ? DrCfg<128>::TEAMS : a.d == 64 ? DrCfg<64>::TEAMS : DrCfg<16>::TEAMS) + 1ll;
    const int all = (int)std::min<long long>(a.n + 1, room);
    auto seen = [&](int pos) { return (double)(!a.causal ? a.n : a.window > 0 ? std::min(pos, a.window) : pos); };
    auto direct = [&](double L) { return kd * L + c0; };
    auto iterative = [&](double L) { return ks * L + s0; };
    int line = std::max(a.head_rows, 1);
    while (line <= a.n && direct(seen(line)) <= iterative(seen(line))) line += 64;
    if (!a.causal) line = direct(a.n) <= iterative(a.n) ? all : 1;
    if (line > a.n) return all;
    double t_direct = 0.0, t_split = 0.0;                // microseconds of an SM, summed over a head's rows
    for (int r = 0; r < a.nq; r += 32) {
        const int rows = std::min(32, a.nq - r), pos = off + r + rows;
        t_direct += rows * direct(seen(pos));
        t_split += rows * (pos < line ? direct(seen(pos)) : iterative(seen(pos)));
    }
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const double heads = (double)a.B * a.H, longest = block_rows * iterative(seen(a.n));
    const double split = std::max(longest, heads * t_split / sms + 0.3 * longest);
    return split < heads * t_direct / sms ? line : all;
}

// Number of leading rows per head handled directly (causal), or nq / 0 (non-causal).
int head_rows_count(const ForwardArgs& a) {
    const int below = direct_rows_below(a);
    if (below <= 0) return 0;
    if (a.causal) {     // query row i sees n - nq + i + 1 keys
        const int rows = below - 1 - (a.n - a.nq);
        return rows < 0 ? 0 : (rows > a.nq ? a.nq : rows);
    }
    return a.n < below ? a.nq : 0;
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

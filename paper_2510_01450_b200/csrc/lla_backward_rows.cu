// Backward pass of the rows that see fewer than head_rows keys: C is ill-conditioned there (rank-deficient up to the
// ridge), so the whole row -- both solves and every pair term -- runs in fp64 with an explicit C and a direct solve, the
// same split the forward makes.  Notation: header of lla_backward.cu.
//
// The block structure is that of the forward's direct rows (lla_direct_rows.cu): a few consecutive rows of a head, a
// team of warps each, keys and values staged as doubles, every product on the fp64 matrix instruction.  gamma_j and
// the scores come first; then the moments (C's lower block triangle, kbar, sum_j p_j gamma_j k_j), one factorisation with
// the two right-hand sides, e_j and f_j, the per-key coefficients, dQ = t + DS K per row, and
//     dK += DS^T Q + U^T Y + W^T T,   dV += A^T G
// as products over the block's rows, so that a block adds to a gradient entry once instead of once per row.
//
// A row's weights and per-key coefficients stay in shared memory for its up to 2 d keys.  Where the caller raises head_rows
// beyond that (LONG) only the weights and gamma do, in rows as long as needed, and e_j and f_j are formed a chunk of
// keys at a time, e_j once more before for g . o_i.
//
// Measured on B200: 32 heads, n = 1000, d = 64 (95 rows a head) 130 us; 16 heads, d = 128 (191 rows) 1.1 ms.  (One block per
// row with a shared-memory LDL^T on the CUDA cores and one atomic per row and entry: 305 us and 3.5 ms.)
#include "lla_rows.cuh"

namespace lla {
namespace {

template <int D, bool LONG>
struct BrSmem {
    using C = DrCfg<D>;
    static constexpr int LMAX = 2 * D, LDL = LMAX + 4;             // most keys of a row, and a row stride of 4 mod 16
    union {
        double kv[C::CH][C::LDK];
        double mat[C::TEAMS][team::Cfg<D, C::NW>::LOWER][64];
    };
    double q[C::TEAMS][C::LDK], g[C::TEAMS][C::LDK];               // query rows and upstream gradients
    double p[LONG ? 1 : C::TEAMS][LDL];                            // scores -> weights -> a_j              (LONG: these two
    double gam[LONG ? 1 : C::TEAMS][LDL];                          // gamma_j -> scale dL/ds_j               lie behind the struct)
    double kbar[C::TEAMS][D];
    team::Smem<D, C::NW, 2> solve[C::TEAMS];                       // afterwards e_j and f_j lie over its first part
    double red[2][C::TEAMS][C::NW];
    unsigned bad[2];                                               // keys, values at the block's end that are not finite (see Ends)
    int odd;                                                       // a query or upstream gradient of the block is not
    static_assert(64 + D / 8 * 24 + 4 * D >= 2 * LDL, "e and f lie over the solver's w, piv, b and z");
    static_assert(LDL >= C::CH, "e and f of a chunk");
};
// LONG: row stride of the weights and of gamma for rows of up to lmax keys (in whole eights, 4 mod 16 doubles)
__host__ __device__ constexpr int long_stride(int lmax) { return (lmax + 15) / 16 * 16 + 4; }

__device__ __forceinline__ double ld_any(const void* p, int dtype, size_t i) {
    return dtype == LLA_F32 ? (double)static_cast<const float*>(p)[i] : (double)__bfloat162float(static_cast<const __nv_bfloat16*>(p)[i]);
}

template <int D, bool LONG>
__global__ void __launch_bounds__(DrCfg<D>::THREADS, D == 64 && !LONG ? 2 : 1)
bwd_rows_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                const void* __restrict__ dout, int dout_dtype, float* __restrict__ dq, float* __restrict__ dk, float* __restrict__ dv,
                int n, int nq, int rows_per_head, double scale, double lambda, int* __restrict__ status, float* __restrict__ dlambda,
                int H, int kv_group, int lmax) {
    using C = DrCfg<D>;
    using S = BrSmem<D, LONG>;
    using T = team::Cfg<D, C::NW>;
    constexpr int NW = C::NW, TEAMS = C::TEAMS, CH = C::CH, NB = C::NB, R = T::R;
    constexpr unsigned FULL = 0xffffffffu;
    static_assert(C::HALVES == 1, "a warp per eight columns of dQ");
    extern __shared__ __align__(16) unsigned char br_smem[];
    S& sm = *reinterpret_cast<S*>(br_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const int tm = warp / NW, w = warp % NW, tt = tid % (32 * NW);
    const int bar_id = 1 + tm;
    const int bh = blockIdx.x;
    const int i0 = (gridDim.y - 1 - blockIdx.y) * TEAMS;                // rows with the most keys first
    const int i = i0 + tm;
    const bool live = i < rows_per_head;
    const int off = n - nq;
    const int L = live ? off + i + 1 : 0;                               // query row i sits at position off + i
    const int Lb = off + min(i0 + TEAMS, rows_per_head);                // keys of the block
    if (!LLA_IN_BOUNDS(Lb, lmax + 1, status, 602)) return;              // (debug build: the keys must fit the arrays)
    const int ldl = LONG ? long_stride(lmax) : S::LDL, lpad = LONG ? ldl - 4 : S::LMAX;
    double* const ps = LONG ? reinterpret_cast<double*>(br_smem + sizeof(S)) : &sm.p[0][0];
    double* const gams = LONG ? ps + TEAMS * ldl : &sm.gam[0][0];
    auto p_of = [&](int r) { return ps + r * ldl; };
    auto gam_of = [&](int r) { return gams + r * ldl; };
    const size_t base = (size_t)bh * nq;                                // rows of q, dout, dq, dlambda
    const size_t kvbase = (size_t)kv_unit(bh, H, kv_group) * n;         // grouped heads: the key/value head's rows
    const __nv_bfloat16* kb = k + kvbase * D;
    const __nv_bfloat16* vb = v + kvbase * D;
    auto row_of = [](auto& rows) { return [&rows](int r) { return &rows[r][0]; }; };
    auto team_sum = [&](double x, int slot, bool is_max = false) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double z = __shfl_xor_sync(FULL, x, o);
            x = is_max ? fmax(x, z) : x + z;
        }
        if (lane == 0) sm.red[slot][tm][w] = x;
        team::sync<NW>(bar_id);
        x = sm.red[slot][tm][0];
#pragma unroll
        for (int u = 1; u < NW; ++u) x = is_max ? fmax(x, sm.red[slot][tm][u]) : x + sm.red[slot][tm][u];
        return x;
    };
    bool odd = false;
    for (int e = tid; e < TEAMS * D; e += C::THREADS) {
        const int r = e / D, c = e % D;
        const bool in = i0 + r < rows_per_head;
        sm.q[r][c] = in ? (double)__bfloat162float(q[(base + i0 + r) * D + c]) : 0.0;
        sm.g[r][c] = in ? ld_any(dout, dout_dtype, (base + i0 + r) * D + c) : 0.0;
        odd = odd || !isfinite(sm.q[r][c]) || !isfinite(sm.g[r][c]);
    }
    const int L0 = off + i0 + 1;                                         // every row of the block sees the keys before L0
    const Ends ends{L0, Lb, 0, 0};
    odd = __syncthreads_or(odd);
    if (tid == 0) {
        sm.odd = odd;
        sm.bad[0] = sm.bad[1] = 0u;
    }
    auto checked = [&](int j0, int nk, int what) { take_out<D>(sm.kv, L0 - j0, nk, 1u, &sm.bad[what]); };    // (before the barrier that ends the staging)
    // ---- gamma_j = g . v_j and the scores ----
    for (int j0 = 0; j0 < Lb; j0 += CH) {
        const int nk = min(CH, Lb - j0);
        __syncthreads();
        stage<D>(sm.kv, vb, D, j0, Lb, CH);
        checked(j0, nk, 1);
        __syncthreads();
        dots<D>([&](int r) { return gam_of(r) + j0; }, row_of(sm.g), sm.kv, nk, warp, lane);
        __syncthreads();
        stage<D>(sm.kv, kb, D, j0, Lb, CH);
        checked(j0, nk, 0);
        __syncthreads();
        dots<D>([&](int r) { return p_of(r) + j0; }, row_of(sm.q), sm.kv, nk, warp, lane);
    }
    __syncthreads();
    // ---- weights (relative to the row maximum) ----
    double m = -1e300;
    for (int j = tt; j < L; j += 32 * NW) m = fmax(m, p_of(tm)[j] * scale);
    m = team_sum(m, 0, true);
    double omega = 0.0, gsum = 0.0;
    for (int j = tt; j < lpad; j += 32 * NW) {
        const double e = j < L ? exp(p_of(tm)[j] * scale - m) : 0.0;
        omega += e;
        if (j < L) gsum += e * gam_of(tm)[j];
        p_of(tm)[j] = e;
        if (j >= L) gam_of(tm)[j] = 0.0;
    }
    if (sm.bad[0] & ends.seen(tm, 0)) omega = NAN;      // the row sees a key, a value that is not finite
    if (sm.bad[1] & ends.seen(tm, 0)) gsum = NAN;
    omega = team_sum(omega, 1);
    gsum = team_sum(gsum, 0);
    // ---- moments ----
    double c[T::NBLK][2], asum[R], hsum[R];
#pragma unroll
    for (int e = 0; e < T::NBLK; ++e) c[e][0] = c[e][1] = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) asum[r] = hsum[r] = 0.0;
    for (int j0 = 0; j0 < Lb; j0 += CH) {
        if (Lb > CH) {
            __syncthreads();
            stage<D>(sm.kv, kb, D, j0, Lb, CH);
            checked(j0, min(CH, Lb - j0), 0);
            __syncthreads();
        }
        const int ns = (min(CH, L - j0) + 3) / 4;
        team::with_warp<NW>(w, [&](auto wc) {
            constexpr int W = decltype(wc)::value;
#pragma unroll 1
            for (int s = 0; s < ns; ++s) {
                const double* kr = sm.kv[4 * s + t4] + g;
                const double wj = p_of(tm)[j0 + 4 * s + t4], gj = gam_of(tm)[j0 + 4 * s + t4];
                double av[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    av[r] = wj * kr[8 * T::row(r, W)];
                    asum[r] += av[r];
                    hsum[r] += av[r] * gj;
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
    team::Smem<D, NW, 2>& ss = sm.solve[tm];
    const double inv = 1.0 / omega, gbar = gsum * inv, em_om = exp(-m) * inv;      // em_om: d(ridge of C) / d(lambda)
    if (live) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            double a = asum[r], h = hsum[r];
            a += __shfl_xor_sync(FULL, a, 1);
            a += __shfl_xor_sync(FULL, a, 2);
            h += __shfl_xor_sync(FULL, h, 1);
            h += __shfl_xor_sync(FULL, h, 2);
            const int cc = 8 * T::row(r, w) + g;
            if (t4 == 0) {
                sm.kbar[tm][cc] = a * inv;
                ss.b[0][cc] = a * inv - sm.q[tm][cc];
                ss.b[1][cc] = h * inv - gbar * (a * inv);
            }
        }
    }
    __syncthreads();               // the keys are no longer read: their place takes the matrices
    double mb[D / 32] = {};        // kbar - q, entries lane + 32 u
    bool ok = true;
    if (live) {
        const double eps = lambda * em_om;
#pragma unroll
        for (int u = 0; u < D / 32; ++u) mb[u] = sm.kbar[tm][lane + 32 * u] - sm.q[tm][lane + 32 * u];
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
                        if (g == 2 * t4) v0 += eps;
                        if (g == 2 * t4 + 1) v1 += eps;
                    }
                    *reinterpret_cast<double2*>(&sm.mat[tm][team::blk(bi, j)][2 * lane]) = make_double2(v0, v1);
                }
        }
        team::sync<NW>(bar_id);
        ok = team::solve<D, NW, 2>(sm.mat[tm], ss, NB, w, lane, bar_id);
    } else {
        for (int e = tt; e < D; e += 32 * NW) ss.x[0][0][e] = ss.x[0][1][e] = 0.0;
    }
    if (!ok && tt == 0 && status) atomicAdd(status + LLA_STATUS_BAD_PIVOT, 1);
    // y = x[0][0], t = x[0][1].  kbar . y, kbar . t, t . (kbar - q), t . y
    double ky = 0.0, kt = 0.0, tmb = 0.0, ty = 0.0;
    if (live) {
#pragma unroll
        for (int u = 0; u < D / 32; ++u) {
            const int e = lane + 32 * u;
            const double y = ss.x[w][0][e], t = ss.x[w][1][e], kbv = sm.kbar[tm][e];
            ky += kbv * y;
            kt += kbv * t;
            tmb += t * mb[u];
            ty += t * y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ky += __shfl_xor_sync(FULL, ky, o);
            kt += __shfl_xor_sync(FULL, kt, o);
            tmb += __shfl_xor_sync(FULL, tmb, o);
            ty += __shfl_xor_sync(FULL, ty, o);
        }
        if (dlambda && tt == 0) dlambda[base + i] = (float)(em_om * ty);     // dL = t^T dC y
    }
    // ---- e_j = (k_j - kbar) . y, f_j = (k_j - kbar) . t ----
    auto y_of = [&](int r) { return &sm.solve[r].x[0][0][0]; };
    auto t_of = [&](int r) { return &sm.solve[r].x[0][1][0]; };
    auto e_of = [&](int r) { return reinterpret_cast<double*>(&sm.solve[r]); };
    auto f_of = [&](int r) { return reinterpret_cast<double*>(&sm.solve[r]) + S::LDL; };
    // (LONG: of the chunk from e0 on, which lies at the arrays' start)
    auto kappa_of = [&](int from, int to, int e0) {
        double x = 0.0;
        for (int j = from + tt; j < to; j += 32 * NW) x += p_of(tm)[j] * (1.0 - (e_of(tm)[j - e0] - ky)) * gam_of(tm)[j];
        return x;
    };
    double kappa = 0.0;
    for (int j0 = 0; j0 < Lb; j0 += CH) {
        const int nk = min(CH, Lb - j0), at = LONG ? 0 : j0;
        __syncthreads();
        stage<D>(sm.kv, kb, D, j0, Lb, CH);
        checked(j0, nk, 0);
        __syncthreads();
        dots<D>([&](int r) { return e_of(r) + at; }, y_of, sm.kv, nk, warp, lane);
        if constexpr (!LONG) {
            dots<D>([&](int r) { return f_of(r) + at; }, t_of, sm.kv, nk, warp, lane);
        } else {
            __syncthreads();
            kappa += kappa_of(j0, min(L, j0 + nk), j0);
        }
    }
    __syncthreads();
    // ---- per key: a_j -> p, scale dL/ds_j -> gam, p (f - gamma + gbar) -> f, p (e - 1) -> e ----
    if constexpr (!LONG) kappa = kappa_of(0, L, 0);
    kappa = team_sum(kappa, 1) * inv + tmb;                              // g . o_i + t . (kbar - q)
    auto coefficients = [&](int from, int to, int e0) {
        for (int j = from + tt; j < to; j += 32 * NW) {
            double a = 0.0, ds = 0.0, fu = 0.0, ew = 0.0;
            if (j < L) {
                const double p = p_of(tm)[j] * inv, e = e_of(tm)[j - e0] - ky, f = f_of(tm)[j - e0] - kt, gj = gam_of(tm)[j];
                a = p * (1.0 - e);
                ds = scale * p * (gj * (1.0 - e) + (gbar + f) * e - f - kappa);
                fu = p * (f - gj + gbar);
                ew = p * (e - 1.0);
            }
            p_of(tm)[j] = a;
            gam_of(tm)[j] = ds;
            f_of(tm)[j - e0] = fu;
            e_of(tm)[j - e0] = ew;
        }
    };
    if constexpr (!LONG) coefficients(0, S::LMAX, 0);
    // ---- dQ = t + DS K;  dK += DS^T Q + U^T Y + W^T T;  dV += A^T G ----
    double o0 = 0.0, o1 = 0.0;
    const int tr = t4 < TEAMS ? t4 : 0;                                  // A^T operands: row t4 of the block
    const bool tin = t4 < TEAMS;
    for (int j0 = 0; j0 < Lb; j0 += CH) {
        const int nk = min(CH, Lb - j0);
        __syncthreads();
        if (Lb > CH) {
            stage<D>(sm.kv, kb, D, j0, Lb, CH);
            checked(j0, nk, 0);
            __syncthreads();
        }
        const int at = LONG ? j0 : 0;                                    // e and f: their first key
        if constexpr (LONG) {
            dots<D>(e_of, y_of, sm.kv, nk, warp, lane);
            dots<D>(f_of, t_of, sm.kv, nk, warp, lane);
            __syncthreads();
            coefficients(j0, j0 + (nk + 7) / 8 * 8, j0);
            __syncthreads();
        }
        // (warp: columns 8 warp .. + 7)
        for (int s = 0; 4 * s < nk; ++s)
            team::dmma(o0, o1, g < TEAMS ? gam_of(g)[j0 + 4 * s + t4] : 0.0, sm.kv[4 * s + t4][8 * warp + g]);
        const double bq = tin ? sm.q[tr][8 * warp + g] : 0.0, bg = tin ? sm.g[tr][8 * warp + g] : 0.0;
        const double by = tin ? y_of(tr)[8 * warp + g] : 0.0, bt = tin ? t_of(tr)[8 * warp + g] : 0.0;
#pragma unroll 2
        for (int kk = 0; 8 * kk < nk; ++kk) {
            const int j = j0 + 8 * kk + g;                               // (the arrays are zero from L on)
            double x0 = 0.0, x1 = 0.0, z0 = 0.0, z1 = 0.0;
            team::dmma(x0, x1, tin ? gam_of(tr)[j] : 0.0, bq);
            team::dmma(z0, z1, tin ? p_of(tr)[j] : 0.0, bg);
            team::dmma(x0, x1, tin ? f_of(tr)[j - at] : 0.0, by);
            team::dmma(x0, x1, tin ? e_of(tr)[j - at] : 0.0, bt);
            if ((sm.odd || sm.bad[0] || sm.bad[1]) && j >= L0 && j < Lb) {
                // a row that is not finite must not reach the keys that it does not see: only those that do, by hand
                const int c = 8 * warp + 2 * t4;
                x0 = x1 = z0 = z1 = 0.0;
                for (int r = j - L0 + 1; r < min(TEAMS, rows_per_head - i0); ++r) {
                    x0 += gam_of(r)[j] * sm.q[r][c] + f_of(r)[j - at] * y_of(r)[c] + e_of(r)[j - at] * t_of(r)[c];
                    x1 += gam_of(r)[j] * sm.q[r][c + 1] + f_of(r)[j - at] * y_of(r)[c + 1] + e_of(r)[j - at] * t_of(r)[c + 1];
                    z0 += p_of(r)[j] * sm.g[r][c];
                    z1 += p_of(r)[j] * sm.g[r][c + 1];
                }
            }
            if (j < Lb) {
                const size_t at = (kvbase + j) * D + 8 * warp + 2 * t4;
                atomicAdd(reinterpret_cast<float2*>(dk + at), make_float2((float)x0, (float)x1));
                atomicAdd(reinterpret_cast<float2*>(dv + at), make_float2((float)z0, (float)z1));
            }
        }
    }
    if (g < TEAMS && i0 + g < rows_per_head) {
        const double2 t = *reinterpret_cast<const double2*>(t_of(g) + 8 * warp + 2 * t4);
        *reinterpret_cast<float2*>(dq + (base + i0 + g) * D + 8 * warp + 2 * t4) = make_float2((float)(t.x + o0), (float)(t.y + o1));
    }
}

template <int D, bool LONG>
int launch_t(const BackwardArgs& a, int nq, int rows, cudaStream_t stream) {
    using C = DrCfg<D>;
    const int lmax = LONG ? a.n - nq + rows : BrSmem<D, LONG>::LMAX;
    const int smem = (int)(sizeof(BrSmem<D, LONG>) + (LONG ? 2 * sizeof(double) * C::TEAMS * long_stride(lmax) : 0));
    auto kern = bwd_rows_kernel<D, LONG>;
    LLA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    LLA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    dim3 grid(a.B * a.H, (rows + C::TEAMS - 1) / C::TEAMS);
    kern<<<grid, C::THREADS, smem, stream>>>((const __nv_bfloat16*)a.q, (const __nv_bfloat16*)a.k, (const __nv_bfloat16*)a.v, a.dout, a.dout_dtype,
                                             a.dq, a.dk, a.dv, a.n, nq, rows, (double)a.scale, (double)a.lambda, a.status, a.dlambda, a.H,
                                             a.kv_group > 0 ? a.kv_group : 1, lmax);
    LLA_CUDA_TRY(cudaGetLastError());
    return LLA_OK;
}

}  // namespace

int backward_rows_most_keys(int d) { return d == 64 ? 1222 : 323; }

// The first `rows` query rows of every head (they see at most backward_rows_most_keys keys) on `stream`; dK and dV are added to.
int launch_backward_rows(const BackwardArgs& a, int nq, int rows, cudaStream_t stream) {
    const bool many = a.n - nq + rows > 2 * a.d;
    if (a.d == 64) return many ? launch_t<64, true>(a, nq, rows, stream) : launch_t<64, false>(a, nq, rows, stream);
    if (a.d == 128) return many ? launch_t<128, true>(a, nq, rows, stream) : launch_t<128, false>(a, nq, rows, stream);
    return LLA_ERR_UNSUPPORTED;
}

}  // namespace lla

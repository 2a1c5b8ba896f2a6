// LLA decode on tensor cores (bf16 caches, d = dv = 64 or 128): one pass over the KV cache.
//
// The cache is streamed a single time and folded into the weighted moments about the origin that the
// centred form of Eq. "lla_decomp" needs:
//     M = sum_j w_j k_j k_j^T,  N = sum_j w_j v_j k_j^T  (fp32 in TMEM),  omega = sum w (CUDA cores),
//     a = sum w k,  c = sum w v  (d = 64: a column of the MMA; d = 128: CUDA cores).
//
// Per tile of 64 keys, each role at its own pace, coupled by mbarriers only:
//   TMA         K and V tiles -> 128B-swizzled shared memory, where they are the MN-major B operand as they arrive:
//               nothing is written to shared memory by a thread except the weights.
//   4 or 8 warps  scores and weights (d / 32 lanes per key), weights to shared memory; omega (and c at d = 128)
//   4 or 8 warps  the A operand: a key (or value) tile is read transposed (ldmatrix.trans), scaled by the weights and
//               stored to TMEM as bf16 hi + lo (16 to 17 mantissa bits).  The fragment that ldmatrix.trans leaves in a
//               thread -- feature lane / 4, keys 2 (lane % 4), + 1 -- is the one that tcgen05.st.16x128b stores, and the
//               products are formed on those packed pairs.
//   MMA (TS)    d = 64 : A = [wK ; wV]^T (128 rows), B = [K | 1] (N = 80):  D = [M a ; N c]
//               d = 128: A = [wK]^T,                 B = [K | V] (N = 256): D = [M | N^T]; a, c on the CUDA cores
//
// Why this form: [K^T ; V^T] as A and the weighted keys as B, written to shared memory by the threads, take 80 KB of
// shared-memory traffic per 16 KB of cache and one chain of dependent phases per tile (265 us at 64 sequences x 16
// heads, d = 64).  Here it is 56 KB and the phases of different tiles overlap (230 us).
//
// Precision: the accumulators are fp32, added to once per 16 keys and operand half.  Against float64 the output at
// d = 128 differs by 4e-6 (500 keys a part) to 3e-5 (8000), which grows with the number of these additions, not with the
// operands' 17 bits; at d = 64 by the solve's tolerance, 5e-5.  The CUDA-core kernels (impl = LLA_IMPL_SIMT) give 1e-6.
//
// m_ref is the maximum of the first tile.  The threads only note whether a later score exceeds it by more
// than 2^90 (no check per tile across threads); if one did, the whole pass is repeated with the true maximum, which
// is known by then (never triggered by bounded scores, covered by a test).  After the last tile the moments go to
// the workspace as a record for the solve kernel, or, without one, to shared memory and are solved on the spot.
#include "lla_sm100.cuh"

namespace lla {
namespace {

using namespace sm100;

constexpr int DT_MAX_RANKED = 1024;   // batches up to this size are processed longest-first
constexpr int DT_BK = 64;             // keys per tile

template <int D>
struct DtCfg {
    static constexpr int NSUB = D / 64;                    // 64-column sub-tiles of K (and of V) in a stage
    static constexpr int SUB = DT_BK * 128;                // bytes of a sub-tile
    static constexpr int STAGE = 2 * NSUB * SUB;           // K tile, V tile
    static constexpr int NST = D == 64 ? 5 : 6;            // ring stages: 80 KB and two blocks per SM at d = 64, 192 KB and one at d = 128
    static constexpr int NMMA = D == 64 ? 80 : 256;        // accumulator columns (d = 64: a ones column at 64, padded to 16)
    static constexpr int TC_A = D == 64 ? 96 : 256;        // first TMEM column of the A operand buffers
    static constexpr int NAB = D == 64 ? 2 : 4;            // these buffers, 64 columns each (hi 32, lo 32)
    static constexpr int TMEM = D == 64 ? 256 : 512;
    static_assert(TC_A + 64 * NAB <= TMEM, "TMEM");
    static constexpr uint32_t IDESC = make_idesc(128, NMMA, 0, 1);
    static constexpr int NBG = D / 64;                     // groups of four score warps and of four operand warps, which
    static constexpr int NSW = 4 * NBG;                    // take the tiles in turn
    static constexpr int KPP = 1024 / D;                   // keys of a score warp and pass (d / 32 lanes per key)
    static constexpr int PASSES = 16 / KPP;                // passes over the 16 keys of a score warp
    static constexpr int W_TMA = NSW + 4 * NBG;            // warps: scores, operand, TMA, MMA
    static constexpr int THREADS = 32 * (W_TMA + 2);
    static constexpr int REC = 2 * D * D + 2 * D + 4;      // floats of a moment record: M, N^T, a, c, omega, m, 2 pad
    static constexpr int SM_ONES = NST * STAGE;            // d = 64: a tile of 64 rows whose column 0 is 1 and the rest 0
    static constexpr int SM_BAR = SM_ONES + (D == 64 ? SUB : 0);
    static constexpr int SM_MISC = SM_BAR + 256;           // tmem base, abort, repeat flag, warp maxima
    static constexpr int SM_W = SM_MISC + 128;             // NST x 64 weights as bf16 pairs: per two keys hi, hi, lo, lo
    static constexpr int SM_WF = SM_W + NST * DT_BK * 4;   // NST x 64 weights, fp32
    static constexpr int SM_TOTAL = SM_WF + (D == 128 ? NST * DT_BK * 4 : 0);
    static constexpr int SM_ALLOC = SM_TOTAL + 1024;
    enum { KVFULL = 0, KVEMPTY = KVFULL + NST, WFULL = KVEMPTY + NST, AFULL = WFULL + NST, AFREE = AFULL + NAB,
           DFULL = AFREE + NAB, PASS = DFULL + 2, EXIT = PASS + 1, NBAR = EXIT + 1 };
    static_assert(NBAR * 8 <= 256, "barrier area too small");
};

// D += A_hi B, D += A_lo B over 64 keys.  B is MN-major, 128B swizzle: 64-column groups one sub-tile apart (leading
// byte offset), 8-key groups 1024 bytes apart; a 16-key step is 2048 bytes (128 descriptor units) and 8 columns of A.
// At d = 64 the second column group is the ones tile, so that column 64 of D is the row sum of the operand.
template <int D>
__device__ __forceinline__ void mma_tile(uint32_t el, uint32_t d, uint32_t a, uint32_t kv_smem, uint32_t ones, bool first) {
    using C = DtCfg<D>;
    const uint64_t b = make_desc(kv_smem, D == 64 ? ones - kv_smem : (uint32_t)C::SUB);
    mma_ts_k64c(el, d, a, b, C::IDESC, first ? 0u : 1u);
    mma_ts_k64c(el, d, a + 32, b, C::IDESC, 1u);
}

// packed bf16 arithmetic
__device__ __forceinline__ uint32_t mul_bf2(uint32_t a, uint32_t b) { uint32_t r; asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ uint32_t fma_bf2(uint32_t a, uint32_t b, uint32_t c) { uint32_t r; asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c)); return r; }
// four 8 x 8 blocks of 16-bit elements, each transposed: lane l gets row l / 4, columns 2 (l % 4) and + 1 of every block
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}
// 16 TMEM lanes x 16 columns: r[2 g] is lane l / 4 and r[2 g + 1] lane l / 4 + 8, column 4 g + l % 4
__device__ __forceinline__ void tmem_st_16x128(uint32_t addr, const uint32_t (&r)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
        ::"r"(addr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}

// ------------------------------------------------------------------------------------------------
// The d x d solve of one (sequence, head), by d threads
// ------------------------------------------------------------------------------------------------
// C y = q - kbar with C = M / omega - kbar kbar^T + ridge I.  A dense factorisation is a chain of d dependent column
// steps; conjugate gradients need one or two dozen short matrix-vector products instead.  Thread r keeps row r of C
// in registers as fp32 pairs and reads the vector from shared memory as broadcasts, so a product has no shuffles at
// all.  The iteration runs in fp32 on a residual that is formed in fp64 from the records: x += (approximate)
// C^-1 r, r = b - C x, until |r| <= tol |b| holds for the fp64 residual.  Usually one round (tol 1e-4) or two (1e-6).
// The recurrences are the Chronopoulos-Gear form: both inner products of an iteration, (r, r) and (C r, r), are taken
// after the matrix-vector product, so an iteration has one reduction and two barriers.
template <int D>
struct SvCfg {
    static constexpr int NW = D / 32;                // warps
    static constexpr int CAP = 3 * D;                // CG iterations in all (the elimination takes over beyond it)
    // Relative residual.  d = 64: the forward's own CG tolerance for bf16 inputs; the output error is then 1.1e-4
    // row-wise, as for a prefill row (1e-5 gives 1.6e-5, 1e-9 0.8e-5 -- from there on the fp32 moments set it).
    // d = 128: where the error of the fp32 moments stands.
    static constexpr double TOL = D == 64 ? 1e-4 : 1e-6;
};
template <int D>
struct alignas(16) SolveSmem {
    float p[D];                              // vector of the current product, fp32
    float red[2][2 * SvCfg<D>::NW];
    double dred[2 * SvCfg<D>::NW];
    double a[D], c[D], x[D];                 // kbar, vbar, solution
};
template <int D>
__device__ __forceinline__ void sv_sync() { asm volatile("bar.sync 2, %0;" ::"n"(D) : "memory"); }

template <int D>
__device__ __forceinline__ double sv_sum(double v, SolveSmem<D>& sm) {
    const int tid = threadIdx.x;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    sv_sync<D>();
    if ((tid & 31) == 0) sm.dred[tid >> 5] = v;
    sv_sync<D>();
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < SvCfg<D>::NW; ++i) s += sm.dred[i];
    return s;
}

// Gaussian elimination without pivoting in fp64 (the matrix is symmetric positive definite), thread r on row r; only
// for systems on which the conjugate gradients gave up.  Returns false if a pivot was not positive.
template <int D>
__device__ __noinline__ bool sv_eliminate(const float* src, double inv, double ridge, double b, SolveSmem<D>& sm, double* prow) {
    const int r = threadIdx.x;
    double row[D];
    for (int j = 0; j < D; ++j) row[j] = (double)src[j * D + r] * inv - sm.a[j] * sm.a[r] + (j == r ? ridge : 0.0);
    bool ok = true;
    for (int k = 0; k < D; ++k) {
        sv_sync<D>();
        if (r == k) {
            for (int j = k; j < D; ++j) prow[j] = row[j];
            prow[D] = b;
        }
        sv_sync<D>();
        const double piv = prow[k];
        if (!(piv > 0.0)) ok = false;
        if (r > k) {
            const double l = row[k] / piv;
            for (int j = k + 1; j < D; ++j) row[j] -= l * prow[j];
            b -= l * prow[D];
        }
    }
    for (int k = D - 1; k >= 0; --k) {
        if (r == k) sm.x[k] = b / row[k];
        sv_sync<D>();
        if (r < k) b -= row[k] * sm.x[k];
    }
    sv_sync<D>();
    return ok;
}

// Centre the moments of one unit at src (global or shared memory), solve and emit the output row.  With several parts
// the matrices and first moments at src are already the sums over the parts (decode_merge_kernel), relative to the
// largest of the parts' maxima; weight and maximum are still those of each part.  Called by threads 0 .. D - 1 of a block.
template <int D, typename TOut>
__device__ __forceinline__ void solve_unit(const __nv_bfloat16* __restrict__ qrow, const float* __restrict__ src, int splits, float lambda_u,
                                           int ridge_mode, TOut* __restrict__ orow, int* __restrict__ status, SolveSmem<D>& sm, double* prow,
                                           float* ms) {
    using C = SvCfg<D>;
    constexpr int PF = DtCfg<D>::REC, NW = C::NW;
    const int r = threadIdx.x, lane = r & 31, wp = r >> 5;
    // ms: shared memory for the second moments, which are on their way while the weights of the parts are looked at, and
    // which the residuals read again (null: src is in shared memory itself)
    if (ms) {
#pragma unroll
        for (int c = 0; c < D / 4; ++c)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(ms + 4 * (c * D + r))), "l"(src + 4 * (c * D + r)) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // weights of the parts: every warp finds the maximum, one lane per part and pass
    float m = -INFINITY;
    for (int p = lane; p < splits; p += 32) m = fmaxf(m, src[(size_t)p * PF + 2 * D * D + 2 * D + 1]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    double omega = 0.0;
    for (int p = lane; p < splits; p += 32)       // (NaN in the record of an aborted block)
        omega += (double)expf(src[(size_t)p * PF + 2 * D * D + 2 * D + 1] - m) * (double)src[(size_t)p * PF + 2 * D * D + 2 * D];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) omega += __shfl_xor_sync(0xffffffffu, omega, off);
    const double inv = 1.0 / omega;
    const double lam_u = (double)lambda_u;
    const double ridge = (ridge_mode == LLA_RIDGE_PRINTED ? lam_u : lam_u * exp(-(double)m)) * inv;
    const double ar = (double)src[2 * D * D + r] * inv, cb = (double)src[2 * D * D + D + r] * inv;
    sm.a[r] = ar;
    sm.x[r] = 0.0;      // the solution where the right-hand side is zero and no round runs
    if (ms) asm volatile("cp.async.wait_group 0;" ::: "memory");
    sv_sync<D>();
    // row r of the centred matrix (column r of the moments: M is symmetric up to fp32 rounding)
    const float* mcol = ms ? ms + r : src + r;
    uint64_t row[D / 2];
#pragma unroll
    for (int j = 0; j < D; j += 8) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = mcol[(j + e) * D];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            double s0 = (double)v[e] * inv - sm.a[j + e] * ar, s1 = (double)v[e + 1] * inv - sm.a[j + e + 1] * ar;
            if (j + e == r) s0 += ridge;
            if (j + e + 1 == r) s1 += ridge;
            row[(j + e) / 2] = pk2((float)s0, (float)s1);
        }
    }
    const double b = (double)to_f32(qrow[r]) - ar;
    double x = 0.0, res = b;
    const double bb = sv_sum<D>(b * b, sm);
    double rr = bb;
    const double stop_all = C::TOL * C::TOL * bb;
    int its = 0;
    bool done = !(bb > 0.0);
    for (int round = 0; round < 6 && !done; ++round) {
        // fp32 conjugate gradients on C e = res, scaled to |res| = 1.  A round reduces the residual by 1e4 at most
        // (what fp32 resolves on these systems), or by what is missing.
        const double scale = rsqrt(rr);
        const float stop = fmaxf(0.81e-8f, (float)(0.81 * stop_all / rr));
        float e = 0.f, rv = (float)(res * scale), pv = 0.f, sv = 0.f, alpha = 0.f, gamma_old = 0.f;
        bool conv = false;
        for (int it = 0; its <= C::CAP; ++it, ++its) {
            sm.p[r] = rv;
            sv_sync<D>();
            const ulonglong2* pp = reinterpret_cast<const ulonglong2*>(sm.p);
            uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
            for (int j = 0; j < D / 4; ++j) {
                const ulonglong2 v = pp[j];
                acc[(2 * j) & 3] = fma2(row[2 * j], v.x, acc[(2 * j) & 3]);
                acc[(2 * j + 1) & 3] = fma2(row[2 * j + 1], v.y, acc[(2 * j + 1) & 3]);
            }
            float w0, w1;
            upk2(add2(add2(acc[0], acc[1]), add2(acc[2], acc[3])), w0, w1);
            const float wv = w0 + w1;
            float g = rv * rv, dl = wv * rv;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                g += __shfl_xor_sync(0xffffffffu, g, off);
                dl += __shfl_xor_sync(0xffffffffu, dl, off);
            }
            float* rb = sm.red[it & 1];
            if (lane == 0) { rb[2 * wp] = g; rb[2 * wp + 1] = dl; }
            sv_sync<D>();
            float gamma = 0.f, delta = 0.f;
#pragma unroll
            for (int i = 0; i < NW; ++i) { gamma += rb[2 * i]; delta += rb[2 * i + 1]; }
            if (!(gamma > stop)) { conv = gamma == gamma; break; }
            float beta = 0.f, denom = delta;
            if (it > 0) {
                beta = __fdividef(gamma, gamma_old);
                denom = delta - beta * __fdividef(gamma, alpha);
            }
            if (!(denom > 0.f)) break;
            alpha = __fdividef(gamma, denom);
            pv = rv + beta * pv;
            sv = wv + beta * sv;
            e += alpha * pv;
            rv -= alpha * sv;
            gamma_old = gamma;
        }
        x += (double)e / scale;
        // the residual in fp64
        sv_sync<D>();
        sm.x[r] = x;
        sv_sync<D>();
        double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
        for (int j = 0; j < D; j += 2) {
            s0 += (double)mcol[j * D] * sm.x[j];
            s1 += (double)mcol[(j + 1) * D] * sm.x[j + 1];
        }
        const double ax = sv_sum<D>(ar * x, sm);
        res = b - ((s0 + s1) * inv - ar * ax + ridge * x);
        const double rr2 = sv_sum<D>(res * res, sm);
        done = rr2 <= stop_all;
        if (!conv || !(rr2 < 0.25 * rr)) break;      // no progress
        rr = rr2;
    }
    bool solved = true;
    if (!done) solved = sv_eliminate<D>(src, inv, ridge, b, sm, prow);      // uniform: the decision comes from block-wide sums
    // o_e = vbar_e + sum_f (N[e][f] / omega - vbar_e kbar_f) y_f
    const double yv = done ? x : sm.x[r];
    const double ky = sv_sum<D>(ar * yv, sm);
    double o0 = 0.0, o1 = 0.0;
#pragma unroll 32
    for (int j = 0; j < D; j += 2) {      // (the matrix row's registers are free: 64 loads in flight)
        o0 += (double)src[D * D + j * D + r] * sm.x[j];
        o1 += (double)src[D * D + (j + 1) * D + r] * sm.x[j + 1];
    }
    store_out(orow + r, (float)((o0 + o1) * inv + cb * (1.0 - ky)));
    if (r == 0 && status) {
        atomicAdd(status + LLA_STATUS_ITER_SUM, its);
        if (!solved) atomicAdd(status + LLA_STATUS_BAD_PIVOT, 1);
    }
}

// the same for a record in shared memory, kept out of line so that its registers do not count in the streaming loop
template <int D, typename TOut>
__device__ __noinline__ void solve_here(const __nv_bfloat16* qrow, const float* rec, float lambda_u, int ridge_mode, TOut* orow,
                                        int* status, SolveSmem<D>& sm, double* prow) {
    solve_unit<D>(qrow, rec, 1, lambda_u, ridge_mode, orow, status, sm, prow, nullptr);
}

struct DtParams {
    int B, H, Lmax, splits, head_rows;
    float scale, lambda;
    const int* lens;
    float* parts;        // moment records; null: solve in the epilogue (one part)
    int* status;
    const float* lambda_units;   // optional per-(sequence, head) ridge
    int ridge_mode;
    int kv_group;        // query heads per key/value head
    int window;          // sliding window (0: none)
    long long wait_clocks;   // cap of every bounded wait, in SM clocks
    int no_loads;        // test aid: the TMA warp issues no copy at all, so that every wait expires with nothing in flight
    PagedKv paged;       // table != nullptr: the tensor maps cover [num_pages * kv heads][page_size][d]
};

template <int D, typename TOut>
__global__ void __launch_bounds__(DtCfg<D>::THREADS, D == 64 ? 2 : 1)
decode_tc_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                 const __nv_bfloat16* __restrict__ q, TOut* __restrict__ out, const DtParams prm) {
    using C = DtCfg<D>;
    constexpr int BK = DT_BK, NST = C::NST, NAB = C::NAB, NBG = C::NBG, NSW = C::NSW, W_TMA = C::W_TMA, W_MMA = W_TMA + 1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bars = sbase + C::SM_BAR;
    auto bar = [&](int i) { return bars + 8u * i; };
    volatile int* misc = reinterpret_cast<volatile int*>(smem + C::SM_MISC);   // [0] tmem base, [1] abort, [2] repeat the pass
    volatile int* abort_flag = misc + 1;
    volatile float* tmax = reinterpret_cast<volatile float*>(smem + C::SM_MISC + 16);   // 2 x 8 warp maxima
    uint8_t* wbuf = smem + C::SM_W;
    float* wfbuf = reinterpret_cast<float*>(smem + C::SM_WF);
    const long long wcap = prm.wait_clocks;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int part = blockIdx.x;
    // Longest caches first: blocks launch in blockIdx order, so block y takes head (y % H) of the
    // sequence whose length has rank (y / H).  Every block ranks the (few) sequence lengths itself.
    int bh = blockIdx.y;
    if (prm.B <= DT_MAX_RANKED) {
        __shared__ int s_len[DT_MAX_RANKED];
        __shared__ int s_pick;
        for (int b = tid; b < prm.B; b += C::THREADS) s_len[b] = visible_keys(prm.lens[b], prm.Lmax, prm.window);
        __syncthreads();
        const int want = blockIdx.y / prm.H;
        for (int b = tid; b < prm.B; b += C::THREADS) {
            const int lb = s_len[b];
            int rank = 0;
            for (int o = 0; o < prm.B; ++o) rank += (s_len[o] > lb) || (s_len[o] == lb && o < b);
            if (rank == want) s_pick = b;
        }
        __syncthreads();
        bh = s_pick * prm.H + blockIdx.y % prm.H;
    }
    const int kstart = first_visible_key(prm.lens[bh / prm.H], prm.Lmax, prm.window);   // sliding window
    const int L = visible_keys(prm.lens[bh / prm.H], prm.Lmax, prm.window);
    // short caches: solved by the direct fp64 kernel.  (Every way out of this kernel waits for the grid before it: that
    // grid may still run when this one has been launched as its programmatic dependent, and nothing else waits for it.)
    if (L < prm.head_rows) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int chunk = ((L + prm.splits - 1) / prm.splits + BK - 1) / BK * BK;
    const int jbeg = part * chunk, jend = min(L, jbeg + chunk);
    const int ntile = jend > jbeg ? (jend - jbeg + BK - 1) / BK : 0;

    if (tid == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(bar(C::KVFULL + s), 1);
            mbar_init(bar(C::KVEMPTY + s), D == 64 ? 1 : 5);      // d = 128: the score warps read V after the weights
            mbar_init(bar(C::WFULL + s), 4);
        }
        for (int b = 0; b < NAB; ++b) { mbar_init(bar(C::AFULL + b), 4); mbar_init(bar(C::AFREE + b), 1); }
        mbar_init(bar(C::DFULL), 1);              // the accumulator is complete: one barrier per pass
        mbar_init(bar(C::DFULL + 1), 1);
        mbar_init(bar(C::PASS), NSW);
        mbar_init(bar(C::EXIT), 1);
        misc[1] = 0;
        misc[2] = 0;      // set by the score warps when the pass has to be repeated
        fence_barrier_init();
    }
    if (D == 64) {
        // (column 0 of row r is the first element of its chunk 0, which the 128-byte swizzle puts at chunk r % 8)
        for (int e = tid; e < C::SUB / 16; e += C::THREADS) {
            const int row = e >> 3;
            *reinterpret_cast<uint4*>(smem + C::SM_ONES + 16 * e) = make_uint4((e & 7) == (row & 7) ? 0x3F80u : 0u, 0u, 0u, 0u);
        }
        fence_proxy_async();
    }
    if (warp == W_TMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(sbase + C::SM_MISC), "r"(C::TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = (uint32_t)misc[0];

    float omega = 0.f, m_ref = -INFINITY;     // score warps; m_ref in log2 units
    // d = 128 only.  Operand warps: sum of w k for the features 16 g + lane / 4 (+ 8) of this warp's lanes, even and odd
    // keys apart; score warps: sum of w v for the eight features of this thread's chunk
    uint64_t sums[2][2] = {{0ull, 0ull}, {0ull, 0ull}};

    if (warp == W_TMA) {
        // ================================ TMA producer ================================
        if (lane == 0 && !prm.no_loads) {
            // K/V unit and row of a tile in the tensor map: (batch, key/value head) and the key index, or for a
            // paged cache (page, key/value head) and the row inside the page (a tile never straddles a page)
            const int hkv = prm.H / prm.kv_group, kvl = (bh % prm.H) / prm.kv_group;
            const int kvh = (bh / prm.H) * hkv + kvl;
            const int* table = prm.paged.table ? prm.paged.table + (size_t)(bh / prm.H) * prm.paged.max_pages : nullptr;
            int issued = 0;      // tiles whose copies have been issued
            for (int g = 0, pass = 0; pass < 2; ++pass) {
              bool okp = true;
              for (int t = 0; t < ntile; ++t, ++g) {      // g: running tile count over both passes (ring position)
                const uint32_t s = g % NST;
                if (!mbar_wait(bar(C::KVEMPTY + s), ((g / NST) & 1) ^ 1, abort_flag, wcap)) { okp = false; break; }
                issued = g + 1;
                const uint32_t dst = sbase + s * C::STAGE;
                mbar_expect_tx(bar(C::KVFULL + s), C::STAGE);
                int unit = kvh, jrow = kstart + jbeg + t * BK;
                if (table) {
                    const int page = min(max(table[jrow / prm.paged.page_size], 0), prm.paged.num_pages - 1);
                    unit = page * hkv + kvl;
                    jrow %= prm.paged.page_size;
                }
#pragma unroll
                for (int sub = 0; sub < C::NSUB; ++sub) {
                    tma_load_3d(dst + sub * C::SUB, &tmK, bar(C::KVFULL + s), 64 * sub, jrow, unit);
                    tma_load_3d(dst + (C::NSUB + sub) * C::SUB, &tmV, bar(C::KVFULL + s), 64 * sub, jrow, unit);
                }
              }
              // a second pass only if the score warps ask for it
              if (!okp || pass == 1 || ntile == 0 || !mbar_wait(bar(C::PASS), 0, abort_flag, wcap) || misc[2] == 0) break;
            }
            if (*abort_flag) {      // an aborted block: the copies issued above must have landed before the block exits
                for (int g = max(0, issued - NST); g < issued; ++g)
                    (void)mbar_wait_landed(bar(C::KVFULL + g % NST), (g / NST) & 1, wcap);
            }
        }
    } else if (warp == W_MMA) {
        // ================================ MMA issuer (whole warp, predicated) ================================
        const uint32_t el = elect_one();
        for (int g = 0, pass = 0; pass < 2; ++pass) {
            bool okp = true;
            for (int t = 0; t < ntile; ++t, ++g) {
                const uint32_t s = g % NST, b = g % NAB;
                if (!mbar_wait(bar(C::KVFULL + s), (g / NST) & 1, abort_flag, wcap)) { okp = false; break; }
                if (!mbar_wait(bar(C::AFULL + b), (g / NAB) & 1, abort_flag, wcap)) { okp = false; break; }
                tc_fence_after();
                mma_tile<D>(el, tmem, tmem + C::TC_A + 64 * b, sbase + s * C::STAGE, sbase + C::SM_ONES, t == 0);     // t == 0 overwrites
                tc_commit_el(el, bar(C::KVEMPTY + s));
                tc_commit_el(el, bar(C::AFREE + b));
                if (t == ntile - 1) tc_commit_el(el, bar(C::DFULL + pass));
            }
            if (!okp || pass == 1 || ntile == 0 || !mbar_wait(bar(C::PASS), 0, abort_flag, wcap) || misc[2] == 0) break;
        }
        if (*abort_flag) {      // an aborted block: the MMAs issued above must be done before TMEM and shared memory go
            tc_commit_el(el, bar(C::EXIT));
            (void)mbar_wait_landed(bar(C::EXIT), 0, wcap);
        }
    } else if (warp < NSW) {
        // ================================ score warps ================================
        // Keys j, j + KPP of the tile, features 32 h .. 32 h + 31.  The eight lanes that share a 128-byte shared-memory
        // wavefront have the same h and neighbouring keys, so the swizzled chunks never collide.
        constexpr int KPP = C::KPP, PASSES = C::PASSES, CH = D / 8;
        const int grp = warp >> 2, h = lane / KPP, j = (warp & 3) * 16 + lane % KPP;
        const uint32_t krow = (h >> 1) * C::SUB + j * 128;
        const float c1 = prm.scale * 1.4426950408889634f;
        uint64_t qv[16];
        {
            const __nv_bfloat16* qp = q + (size_t)bh * D + 32 * h;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float qf[8];
                load8(qp + 8 * i, qf);
#pragma unroll
                for (int e = 0; e < 4; ++e) qv[4 * i + e] = pk2(qf[2 * e] * c1, qf[2 * e + 1] * c1);
            }
        }
        bool ok = true;
        float run_max = -INFINITY, s2[PASSES];
        bool over = false, valid[PASSES];
        // (t: tile of the pass, it fixes the keys; g: running tile count over both passes, it fixes ring stage,
        //  buffer and barrier phase)
        auto score = [&](int t, int g) -> bool {
            const int sl = g % NST;
            const bool landed = mbar_wait(bar(C::KVFULL + sl), (g / NST) & 1, abort_flag, wcap);
            if (!__all_sync(0xffffffffu, landed)) return false;      // what follows is warp-wide
            uint8_t* ks = smem + sl * C::STAGE + krow;
            uint64_t sd[PASSES][4 / PASSES];                          // four independent chains of pairs
#pragma unroll
            for (int u = 0; u < PASSES; ++u)
#pragma unroll
                for (int e = 0; e < 4 / PASSES; ++e) sd[u][e] = 0ull;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < PASSES; ++u) {
                    const uint4 raw = *reinterpret_cast<const uint4*>(ks + u * KPP * 128 + (((4 * (h & 1) + i) ^ (j & 7)) << 4));
                    const uint32_t wds[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint64_t& d = sd[u][e % (4 / PASSES)];
                        d = fma2(qv[4 * i + e], pk2(__uint_as_float(wds[e] << 16), __uint_as_float(wds[e] & 0xFFFF0000u)), d);
                    }
                }
#pragma unroll
            for (int u = 0; u < PASSES; ++u) {
                uint64_t d = sd[u][0];
#pragma unroll
                for (int e = 1; e < 4 / PASSES; ++e) d = add2(d, sd[u][e]);
                float a0, a1;
                upk2(d, a0, a1);
                s2[u] = a0 + a1;
            }
#pragma unroll
            for (int off = KPP; off < 32; off <<= 1)
#pragma unroll
                for (int u = 0; u < PASSES; ++u) s2[u] += __shfl_xor_sync(0xffffffffu, s2[u], off);
#pragma unroll
            for (int u = 0; u < PASSES; ++u) {
                valid[u] = jbeg + t * BK + j + u * KPP < jend;
                if (!valid[u]) s2[u] = -INFINITY;
            }
            if (jbeg + (t + 1) * BK > jend) {
                // ragged last tile: rows past the end may hold anything (unused cache slots).  They are
                // operands, so clear them (0 x NaN would poison the accumulator).
#pragma unroll
                for (int u = 0; u < PASSES; ++u)
                    if (!valid[u]) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t off = u * KPP * 128 + (((4 * (h & 1) + i) ^ (j & 7)) << 4);
                            *reinterpret_cast<uint4*>(ks + off) = make_uint4(0, 0, 0, 0);
                            *reinterpret_cast<uint4*>(ks + C::NSUB * C::SUB + off) = make_uint4(0, 0, 0, 0);
                        }
                    }
                fence_proxy_async();
            }
            return true;
        };
        auto warp_max = [&](float v) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
            return v;
        };
        // The reference maximum is the first tile's; later tiles only note, per thread and without any barrier, the
        // largest score seen and whether one exceeded the reference by more than 2^90 -- then the weights of this pass
        // are useless (they are clamped, so nothing overflows) and the pass is repeated with the true maximum as
        // reference.
        if (ntile > 0) {
            if (grp == 0) {
                ok = score(0, 0);
                float v = s2[0];
#pragma unroll
                for (int u = 1; u < PASSES; ++u) v = fmaxf(v, s2[u]);
                v = warp_max(v);
                if (lane == 0) tmax[warp] = v;
            }
            ok = !bar_or(1, 32 * NSW, !ok);
            m_ref = fmaxf(fmaxf(tmax[0], tmax[1]), fmaxf(tmax[2], tmax[3]));
        }
        for (int pass = 0, g0 = 0; pass < 2 && ntile > 0; ++pass, g0 += ntile) {
            omega = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) sums[i >> 1][i & 1] = 0ull;
            for (int t = grp; t < ntile && ok; t += NBG) {
                const int g = g0 + t, sl = g % NST;
                ok = score(t, g);
                if (!ok) break;
#pragma unroll
                for (int u = 0; u < PASSES; ++u) {
                    run_max = fmaxf(run_max, s2[u]);
                    over |= s2[u] > m_ref + 90.f;
                    const float w = valid[u] ? ex2f(fminf(s2[u] - m_ref, 100.f)) : 0.f;
                    if (h == 0) {
                        omega += w;
                        const int key = j + u * KPP;
                        const __nv_bfloat16 whi = __float2bfloat16_rn(w);
                        const __nv_bfloat16 wlo = __float2bfloat16_rn(w - __bfloat162float(whi));
                        __nv_bfloat16* wj = reinterpret_cast<__nv_bfloat16*>(wbuf + sl * BK * 4 + (key >> 1) * 8) + (key & 1);
                        wj[0] = whi;
                        wj[2] = wlo;
                        if (D == 128) wfbuf[sl * BK + key] = w;
                    }
                }
                // one arrival per warp: 32 lanes arriving on one mbarrier are 32 serialised shared-memory atomics
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(C::WFULL + sl));
                if constexpr (D == 128) {
                    const int vchunk = lane % CH;
                    const uint8_t* vs = smem + sl * C::STAGE + (C::NSUB + (vchunk >> 3)) * C::SUB;
                    const float* wt = wfbuf + sl * BK;
#pragma unroll
                    for (int i = 0; i < 16 * CH / 32; ++i) {
                        const int key = (warp & 3) * 16 + lane / CH + 32 / CH * i;
                        const uint4 x = *reinterpret_cast<const uint4*>(vs + key * 128 + (((vchunk & 7) ^ (key & 7)) << 4));
                        const float w = wt[key];
                        const uint64_t w2 = pk2(w, w);
                        sums[0][0] = fma2(w2, pk2(__uint_as_float(x.x << 16), __uint_as_float(x.x & 0xFFFF0000u)), sums[0][0]);
                        sums[0][1] = fma2(w2, pk2(__uint_as_float(x.y << 16), __uint_as_float(x.y & 0xFFFF0000u)), sums[0][1]);
                        sums[1][0] = fma2(w2, pk2(__uint_as_float(x.z << 16), __uint_as_float(x.z & 0xFFFF0000u)), sums[1][0]);
                        sums[1][1] = fma2(w2, pk2(__uint_as_float(x.w << 16), __uint_as_float(x.w & 0xFFFF0000u)), sums[1][1]);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(C::KVEMPTY + sl));
                }
            }
            // end of a pass.  (A warp whose wait failed still takes part in the barriers; all warps leave together.)
            if (bar_or(1, 32 * NSW, !ok) || pass == 1) break;
            // did any score leave the range of the reference?  (one barrier per pass)
            const bool any = bar_or(1, 32 * NSW, over);
            if (tid == 0) misc[2] = (int)any;
            if (any) {
                const float v = warp_max(run_max);
                if (lane == 0) tmax[8 + warp] = v;
            }
            asm volatile("bar.sync 1, %0;" ::"n"(32 * NSW) : "memory");
            if (any) {
                m_ref = tmax[8];
#pragma unroll
                for (int i = 1; i < NSW; ++i) m_ref = fmaxf(m_ref, tmax[8 + i]);
                over = false;
            }
            if (lane == 0) mbar_arrive(bar(C::PASS));      // the other warps read misc[2] after this
            if (!any) break;
        }
        // total weight of this part
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) omega += __shfl_xor_sync(0xffffffffu, omega, off);
    } else {
        // ================================ operand warps ================================
        // Warp w stores to TMEM lanes 32 (w % 4) .. + 31.  d = 128: the features of that number of the keys; d = 64: lanes
        // 0 .. 63 the keys' features, 64 .. 127 the values'.  The groups of four warps take the tiles in turn.
        const int quad = warp & 3, grp = (warp - NSW) >> 2;
        const uint32_t src0 = D == 64 ? (quad >> 1) * C::NSUB * C::SUB : (quad >> 1) * C::SUB;
        // ldmatrix: lanes 8 m .. 8 m + 7 address matrix m; matrices (key group, chunk), (same, chunk + 1), (next, ..)
        const uint32_t lrow = 8 * (lane >> 4) + (lane & 7);
        const uint32_t lchunk = 4 * (quad & 1) + ((lane >> 3) & 1);
        const uint32_t lane_addr = tmem + ((uint32_t)(32 * quad) << 16) + C::TC_A;
        for (int pass = 0, g0 = 0; pass < 2 && ntile > 0; ++pass, g0 += ntile) {
            bool ok = true;
#pragma unroll
            for (int i = 0; i < 4; ++i) sums[i >> 1][i & 1] = 0ull;
            for (int t = grp; t < ntile; t += NBG) {
                const int g = g0 + t, sl = g % NST, b = g % NAB;
                // the weights and the tile; the operand buffer, released by the MMA of the tile NAB before
                ok = mbar_wait(bar(C::AFREE + b), ((g / NAB) & 1) ^ 1, abort_flag, wcap) &&
                     mbar_wait(bar(C::KVFULL + sl), (g / NST) & 1, abort_flag, wcap) &&
                     mbar_wait(bar(C::WFULL + sl), (g / NST) & 1, abort_flag, wcap);
                ok = __all_sync(0xffffffffu, ok);           // what follows is warp-wide
                if (!ok) break;
                tc_fence_after();
                const uint32_t tile = sbase + sl * C::STAGE + src0 + lrow * 128;
                const uint8_t* wp = wbuf + sl * BK * 4 + 8 * (lane & 3);
                const float* wt = wfbuf + sl * BK + 2 * (lane & 3);
#pragma unroll
                for (int kh = 0; kh < 2; ++kh) {                 // 32 keys at a time
                    uint2 ww[4];                                 // the weights of keys 8 kg + 2 (lane % 4), + 1: hi pair, lo pair
#pragma unroll
                    for (int kg = 0; kg < 4; ++kg) ww[kg] = *reinterpret_cast<const uint2*>(wp + 32 * (4 * kh + kg));
#pragma unroll
                    for (int fg = 0; fg < 2; ++fg) {             // 16 features at a time
                        const uint32_t base = tile + (((lchunk + 2 * fg) ^ (lane & 7)) << 4) + 4096 * kh;
                        uint32_t r[8], lo[8];
#pragma unroll
                        for (int kg = 0; kg < 4; kg += 2) ldsm4_t(base + kg * 1024, r[2 * kg], r[2 * kg + 1], r[2 * kg + 2], r[2 * kg + 3]);
                        if constexpr (D == 128) {
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                sums[fg][i & 1] = fma2(*reinterpret_cast<const uint64_t*>(wt + 32 * kh + 8 * (i >> 1)),
                                                       pk2(__uint_as_float(r[i] << 16), __uint_as_float(r[i] & 0xFFFF0000u)), sums[fg][i & 1]);
                        }
                        // w k = (w_hi + w_lo) k with bf16 w_hi, w_lo: hi = round(w_hi k); w_hi k - hi fits bf16 exactly;
                        // lo = round(w_lo k + that).  Relative error of hi + lo about 2^-17, four instructions per two keys.
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const uint32_t hi = mul_bf2(ww[i >> 1].x, r[i]);
                            lo[i] = fma_bf2(ww[i >> 1].y, r[i], fma_bf2(ww[i >> 1].x, r[i], hi ^ 0x80008000u));
                            r[i] = hi;
                        }
                        const uint32_t at = lane_addr + ((uint32_t)(16 * fg) << 16) + 64 * b + 16 * kh;
                        tmem_st_16x128(at, r);
                        tmem_st_16x128(at + 32, lo);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(C::AFULL + b));
            }
            if (!ok || pass == 1 || !mbar_wait(bar(C::PASS), 0, abort_flag, wcap) || misc[2] == 0) break;
        }
    }

    // ================================ epilogue ================================
    if (warp < W_TMA && ntile > 0) {
        (void)mbar_wait(bar(C::DFULL + (misc[2] ? 1 : 0)), 0, abort_flag, wcap);
        tc_fence_after();
    }
    __shared__ float s_omega[8];
    __shared__ float s_mref;
    if (warp < NSW && lane == 0) s_omega[warp] = omega;
    if (tid == 0) s_mref = m_ref;
    __syncthreads();       // every pipeline stage is drained: shared memory can be re-carved
    const bool aborted = *abort_flag != 0;
    if (aborted) {
        // (the TMA and MMA warps have waited above for what they had issued)
        if (warp == W_TMA) {
            tc_fence_after();
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM) : "memory");
        }
        if (tid == 0) {
            if (prm.status) atomicAdd(prm.status + LLA_STATUS_TIMEOUT, 1);
            if (prm.parts) {
                // no record of this part: poison its weight and maximum, so that the solve kernel emits NaN for the
                // unit instead of reading whatever an earlier call left in the record buffer
                float* dst = prm.parts + ((size_t)bh * prm.splits + part) * C::REC;
                dst[2 * D * D + 2 * D] = __int_as_float(0x7fc00000);
                dst[2 * D * D + 2 * D + 1] = __int_as_float(0x7fc00000);
            }
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    // shared memory now: partial first moments, then (without a workspace) the record
    float* s_fa = reinterpret_cast<float*>(smem);                        // [NBG][128]
    float* s_fc = s_fa + NBG * 128;                                      // [NSW][D]  (d = 128)
    float* s_rec = reinterpret_cast<float*>(smem + 8192);                // REC floats
    if (warp < NSW) {
        if constexpr (D == 128) {
            float cs[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) upk2(sums[i >> 1][i & 1], cs[2 * i], cs[2 * i + 1]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                cs[i] += __shfl_xor_sync(0xffffffffu, cs[i], 16);
                if (lane < 16) s_fc[warp * D + 8 * lane + i] = cs[i];
            }
        }
    } else if (D == 128 && warp < W_TMA) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float e0, e1;
            upk2(sums[i >> 1][i & 1], e0, e1);
            float s = e0 + e1;
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if ((lane & 3) == 0) s_fa[((warp - NSW) >> 2) * 128 + 32 * (warp & 3) + 16 * (i >> 1) + 8 * (i & 1) + (lane >> 2)] = s;
        }
    }
    __syncthreads();
    float omega_tot = 0.f;
#pragma unroll
    for (int i = 0; i < NSW; ++i) omega_tot += s_omega[i];
    const float mref_ln = s_mref * 0.6931471805599453f;          // back to natural-log units
    const bool rec_ok = LLA_IN_BOUNDS((size_t)bh * prm.splits + part, (size_t)gridDim.y * prm.splits, prm.status, 501);
    float* dst = prm.parts ? prm.parts + ((size_t)bh * prm.splits + part) * C::REC : s_rec;
    if (warp < W_TMA && rec_ok) {
        const int quad = warp & 3, cg = warp >> 2;          // TMEM lanes 32 quad .. + 31; columns in 2 or 4 groups
        const int f = 32 * quad + lane;
        constexpr int CPG = D / 2;                            // columns of a group: 32 or 64
        // d = 64: lane f, column c: M[f][c] (f < 64) or N[f - 64][c], stored transposed: both blocks are [c][lane];
        // d = 128: columns 0 .. 127 M[f][c], stored as [c][f]; columns 128 .. 255 N[c - 128][f], stored as [f][c - 128]
#pragma unroll 1
        for (int c0 = CPG * cg; c0 < CPG * cg + CPG; c0 += 32) {
            uint32_t v[32];
            if (ntile > 0) {
                tmem_ld32(tmem + ((uint32_t)(32 * quad) << 16) + c0, v);
                tc_wait_ld();
            } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = 0u;
            }
            if (D == 128 && c0 >= 128) {
#pragma unroll
                for (int e = 0; e < 32; e += 4)
                    *reinterpret_cast<uint4*>(dst + (size_t)D * D + f * D + (c0 - 128) + e) = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
            } else {
                float* p = D == 64 ? dst + (quad >> 1) * D * D + (f & 63) : dst + f;
#pragma unroll
                for (int e = 0; e < 32; ++e) p[(c0 + e) * D] = __uint_as_float(v[e]);
            }
        }
        if (D == 64) {
            if (cg == 0) {                                       // column 64: a then c
                uint32_t v[16] = {0u};
                if (ntile > 0) {
                    tmem_ld16(tmem + ((uint32_t)(32 * quad) << 16) + 64, v);
                    tc_wait_ld();
                }
                dst[2 * D * D + tid] = __uint_as_float(v[0]);
            }
        } else if (tid < D) {
            dst[2 * D * D + tid] = s_fa[tid] + s_fa[(NBG - 1) * 128 + tid];
        } else if (tid < 2 * D) {
            float c = 0.f;
#pragma unroll
            for (int i = 0; i < NSW; ++i) c += s_fc[i * D + tid - D];
            dst[2 * D * D + tid] = c;
        }
        if (tid == 0) {
            dst[2 * D * D + 2 * D] = omega_tot;
            dst[2 * D * D + 2 * D + 1] = ntile > 0 ? mref_ln : -INFINITY;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == W_TMA) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM) : "memory");
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (prm.parts || tid >= D) return;
    // no workspace, one part: solve here
    static_assert(8192 + 4 * C::REC <= C::SM_BAR, "the record does not fit");
    __shared__ SolveSmem<D> sm;
    __shared__ double prow[D + 1];
    solve_here<D>(q + (size_t)bh * D, s_rec, prm.lambda_units ? prm.lambda_units[bh] : prm.lambda, prm.ridge_mode,
                  out + (size_t)bh * D, prm.status, sm, prow);
}

// Sum of the parts' moments of one unit into the record of its first part, each scaled to the largest of their maxima
// (the parts' weights and maxima stay as they are).  Split calls are small ones, which leave most of the chip idle:
// in the solve kernel, whose few blocks would read every part through 64 threads, merging and solving take 42 us at one
// sequence x 16 heads, d = 64, 8 parts; 4 us here and 9 us there.
constexpr int DM_THREADS = 256;
template <int D>
__global__ void __launch_bounds__(DM_THREADS)
decode_merge_kernel(float* __restrict__ parts, const int* __restrict__ lens, int H, int Lmax, int head_rows, int splits, int window) {
    constexpr int PF = DtCfg<D>::REC;
    __shared__ float s_f[kDecodeMaxSplits];
    const int bh = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");      // a programmatic dependent of the streaming kernel
    if (visible_keys(lens[bh / H], Lmax, window) < head_rows) return;
    float* src = parts + (size_t)bh * splits * PF;
    if (tid < 32) {
        float m = -INFINITY;
        for (int p = lane; p < splits; p += 32) m = fmaxf(m, src[(size_t)p * PF + 2 * D * D + 2 * D + 1]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        for (int p = lane; p < splits; p += 32) s_f[p] = expf(src[(size_t)p * PF + 2 * D * D + 2 * D + 1] - m);      // 0 for empty parts
    }
    __syncthreads();
    const int e = blockIdx.x * DM_THREADS + tid;
    if (e >= (2 * D * D + 2 * D) / 4) return;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll 8
    for (int p = 0; p < splits; ++p) {
        const float4 v = reinterpret_cast<const float4*>(src + (size_t)p * PF)[e];
        const double f = (double)s_f[p];
        a0 += f * (double)v.x; a1 += f * (double)v.y; a2 += f * (double)v.z; a3 += f * (double)v.w;
    }
    reinterpret_cast<float4*>(src)[e] = make_float4((float)a0, (float)a1, (float)a2, (float)a3);
}

// Last kernel of the decode with a record buffer.  Several blocks share an SM; the solve is latency-bound (barriers and
// shuffles), which is why it is kept out of the streaming kernel whenever there is a record buffer.
template <int D, typename TOut>
__global__ void __launch_bounds__(D, D == 64 ? 8 : 2)
decode_solve_kernel(const __nv_bfloat16* __restrict__ q, const float* __restrict__ parts, TOut* __restrict__ out,
                    const int* __restrict__ lens, int H, int Lmax, int head_rows, float lambda, int splits,
                    int* __restrict__ status, const float* __restrict__ lambda_units, int ridge_mode, int window) {
    extern __shared__ __align__(16) float sv_mat[];      // D x D
    __shared__ SolveSmem<D> sm;
    __shared__ double prow[D + 1];
    const int bh = blockIdx.x;
    // launched as a programmatic dependent of the streaming kernel: nothing of that grid may be read before this
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (visible_keys(lens[bh / H], Lmax, window) < head_rows) return;
    solve_unit<D>(q + (size_t)bh * D, parts + (size_t)bh * splits * DtCfg<D>::REC, splits, lambda_units ? lambda_units[bh] : lambda,
                  ridge_mode, out + (size_t)bh * D, status, sm, prow, sv_mat);
}

template <int D, typename TOut>
int launch_t(const DecodeArgs& a) {
    using C = DtCfg<D>;
    const int splits = a.splits < 1 ? 1 : a.splits > kDecodeMaxSplits ? kDecodeMaxSplits : a.splits;
    const bool have_ws = decode_records_fit(a);
    if (splits > 1 && !have_ws) return LLA_ERR_WORKSPACE;
    CUtensorMap mk, mv;
    const int BH = a.B * a.H;
    const int kvg = a.kv_group > 0 ? a.kv_group : 1;
    const int map_units = a.paged.table ? a.paged.num_pages * (a.H / kvg) : BH / kvg;
    const int map_rows = a.paged.table ? a.paged.page_size : a.Lmax;
    if (!make_map_bf16(&mk, a.kcache, map_units, map_rows, D, DT_BK) || !make_map_bf16(&mv, a.vcache, map_units, map_rows, D, DT_BK))
        return LLA_ERR_CUDA;
    DtParams prm;
    prm.B = a.B; prm.H = a.H; prm.Lmax = a.Lmax; prm.splits = splits; prm.head_rows = a.head_rows;
    prm.scale = a.scale; prm.lambda = a.lambda; prm.lens = a.lens;
    prm.lambda_units = a.lambda_units; prm.ridge_mode = a.ridge_mode; prm.kv_group = kvg; prm.paged = a.paged; prm.window = a.window;
    prm.wait_clocks = a.wait_clocks > 0 ? a.wait_clocks : kWaitClocks; prm.no_loads = a.no_loads;
    prm.parts = have_ws ? (float*)a.workspace : nullptr; prm.status = a.status;
    // Programmatic dependent launches.  The streaming grid, behind the direct kernel of the short caches (which reads
    // nothing that it writes and writes nothing that it reads), starts as that kernel's blocks leave; the solve grid
    // is set up while the streaming grid drains and its blocks start (past the griddepcontrol.wait at their top) the
    // moment that grid has completed and its records are visible.
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    auto kern = decode_tc_kernel<D, TOut>;
    LLA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SM_ALLOC));
    // two blocks per SM need the largest shared-memory carve-out
    LLA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(splits, BH);
    cfg.blockDim = dim3(C::THREADS);
    cfg.dynamicSmemBytes = C::SM_ALLOC;
    cfg.stream = a.stream;
    cfg.attrs = attr;
    cfg.numAttrs = a.behind_direct ? 1 : 0;
    LLA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, mk, mv, (const __nv_bfloat16*)a.q, (TOut*)a.out, prm));
    if (splits > 1) {
        cudaLaunchConfig_t cm = {};
        cm.gridDim = dim3(((2 * D * D + 2 * D) / 4 + DM_THREADS - 1) / DM_THREADS, BH);
        cm.blockDim = dim3(DM_THREADS);
        cm.stream = a.stream;
        cm.attrs = attr;
        cm.numAttrs = 1;
        LLA_CUDA_TRY(cudaLaunchKernelEx(&cm, decode_merge_kernel<D>, (float*)a.workspace, a.lens, a.H, a.Lmax, a.head_rows, splits, a.window));
    }
    if (have_ws) {
        cudaLaunchConfig_t cs = {};
        cs.gridDim = dim3(BH);
        cs.blockDim = dim3(D);
        cs.dynamicSmemBytes = sizeof(float) * D * D;
        LLA_CUDA_TRY(cudaFuncSetAttribute(decode_solve_kernel<D, TOut>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cs.dynamicSmemBytes));
        LLA_CUDA_TRY(cudaFuncSetAttribute(decode_solve_kernel<D, TOut>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
        cs.stream = a.stream;
        cs.attrs = attr;
        cs.numAttrs = 1;
        LLA_CUDA_TRY(cudaLaunchKernelEx(&cs, decode_solve_kernel<D, TOut>, (const __nv_bfloat16*)a.q, (const float*)a.workspace,
                                        (TOut*)a.out, a.lens, a.H, a.Lmax, a.head_rows, a.lambda, splits, a.status,
                                        a.lambda_units, a.ridge_mode, a.window));
    }
    return LLA_OK;
}

template <int D>
int launch_d(const DecodeArgs& a) {
    if (a.out_dtype == LLA_BF16) return launch_t<D, __nv_bfloat16>(a);
    if (a.out_dtype == LLA_F32) return launch_t<D, float>(a);
    return LLA_ERR_UNSUPPORTED;
}

}  // namespace

// the caller's workspace holds a moment record for every part
bool decode_records_fit(const DecodeArgs& a) {
    return a.workspace && ((uintptr_t)a.workspace & 15u) == 0 && a.workspace_bytes >= decode_record_bytes(a.B, a.H, a.d, a.dv, a.splits);
}

bool decode_tensor_supported(const DecodeArgs& a) {
    return a.in_dtype == LLA_BF16 && a.d == a.dv && (a.d == 64 || a.d == 128) && sm100::get_encode() != nullptr;
}

// Tensor-core decode.  With a record buffer (always for splits > 1, optional for a single part) the streaming kernel writes
// moment records and a solve kernel follows; without one, single-part blocks solve in their own epilogue.
int launch_decode_tensor_moments(const DecodeArgs& a) {
    if (!decode_tensor_supported(a)) return LLA_ERR_UNSUPPORTED;
    return a.d == 64 ? launch_d<64>(a) : launch_d<128>(a);
}

}  // namespace lla

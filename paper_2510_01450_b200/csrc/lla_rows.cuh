// What the kernels of the directly-solved rows share (forward: lla_direct_rows.cu, backward: lla_backward_rows.cu): block
// shapes, staging of keys and values as doubles, and products of a block's rows with the staged keys.
#pragma once

#include "lla_team_solve.cuh"

namespace lla {

template <int D>
struct DrCfg {
    static constexpr int NW = D == 16 ? 1 : D == 64 ? 2 : 8;      // warps per row: what the registers of 16 warps hold
    static constexpr int TEAMS = D == 128 ? 2 : 4;                // rows per block; d = 64: two blocks per SM, so that the pivot
                                                                  // chains of one run beside the products of the other
    static constexpr int WARPS = NW * TEAMS, THREADS = 32 * WARPS;
    // keys per chunk: the keys of a block with a dual row (at most d + TEAMS - 1, with a window d + TEAMS) are one chunk,
    // and at d = 64 so are those of every row solved directly for its few keys
    static constexpr int CH = D == 128 ? 136 : D == 64 ? 128 : 64;
    static constexpr int STEP = D == 128 ? 128 : 64;              // .. and the chunks of longer blocks: eight keys a warp
    static constexpr int LDK = D + 4;                             // row stride in doubles: 4 mod 16, both operand accesses conflict-free
    static constexpr int NB = D / 8;
    static constexpr int HALVES = WARPS / NB;                     // output sum: a warp per 8 columns and part of the keys
    static constexpr int LDW = CH + 4;
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

// keys (or values) j0 .. j0 + ch - 1 -> shared memory; rows from jend on are zero, but the rounds
// that hold no row before jend are left out, four at a time: their rows keep what they held, and nothing reads them.
// (Of rows of 1 to 95 keys, 32 heads, d = 64, all rounds would take 4 % more, forward and backward.)
// REL: ref, a row in shared memory, is subtracted from each of them.
template <int D, bool REL = false, typename TIn>
__device__ __forceinline__ void stage(double (*dst)[DrCfg<D>::LDK], const TIn* __restrict__ src, long long stride, int j0, int jend, int ch,
                                      const double* ref = nullptr) {
    using C = DrCfg<D>;
    constexpr int PER = C::CH * D / 2 / C::THREADS, PER_STEP = C::STEP * D / 2 / C::THREADS;
    static_assert(PER * 2 * C::THREADS == C::CH * D && PER_STEP * 2 * C::THREADS == C::STEP * D, "a chunk is a whole number of rounds");
    constexpr int ROUND = 2 * C::THREADS / D;              // rows of a round
    const int c = 2 * (threadIdx.x % (D / 2));             // the same columns in every round
    const double r0 = REL ? ref[c] : 0.0, r1 = REL ? ref[c + 1] : 0.0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        if (u >= PER_STEP && ch == C::STEP) break;
        if (u % 4 == 0 && j0 + ROUND * u >= jend) break;
        const int j = threadIdx.x / (D / 2) + ROUND * u;
        const bool in = j0 + j < jend;
        double a = 0.0, b = 0.0;
        if (in) load_pair(src + (size_t)(j0 + j) * stride + c, a, b);
        if (REL) {                                         // (outside the condition: the rounds' loads stay together)
            a -= in ? r0 : 0.0;
            b -= in ? r1 : 0.0;
        }
        *reinterpret_cast<double2*>(&dst[j][c]) = make_double2(a, b);
    }
}

// ---- what is not finite ----
// Zero times infinity or NaN is not zero: such entries, in the few keys and values at the ends of a block's range that only
// some of its rows see, would reach the other rows through their zero weights.  They are taken out of the staged rows
// (set to zero; bit b stands for the key hi0 + b, bit 8 + b for lo0 + b), and what the rows that do see them put out is
// spoilt at the end.  (256 fp32 rows, d = 16: 24.6 us with this, 22.5 without; rows of 1 to 95 keys, 32 heads, d = 64: 86 us
// against 84; with bounds on the keys inside the loops over them instead: 24.8 and 86.)
struct Ends {
    int hi0, hi1;      // keys that the last row of the block sees and the first does not: row r sees those before hi0 + r
    int lo0, lo1;      // (window) keys that the first row sees and the last does not
    // the bits of the keys that the block's r-th row sees, if it sees the keys from first_key on
    __device__ __forceinline__ unsigned seen(int r, int first_key) const { return ((1u << r) - 1u) | ((0xff00u << max(first_key - lo0, 0)) & 0xff00u); }
};
// Takes them out of the staged rows first .. first + TEAMS - 2, as far as they are among the nk staged, and notes row first + b as
// bit0 << b in bad.  A thread looks at what it has staged itself, so the barrier that ends the staging is enough.
template <int D>
__device__ __forceinline__ void take_out(double (*rows)[DrCfg<D>::LDK], int first, int nk, unsigned bit0, unsigned* bad) {
    constexpr int ROUND = 2 * DrCfg<D>::THREADS / D;          // a thread stages every ROUND-th row
    static_assert(DrCfg<D>::TEAMS - 1 <= ROUND && (ROUND & (ROUND - 1)) == 0, "at most one of these rows a thread");
    const int b = ((int)threadIdx.x / (D / 2) - first) & (ROUND - 1), j = first + b;
    if (b >= DrCfg<D>::TEAMS - 1 || j < 0 || j >= nk) return;
    double2& x = *reinterpret_cast<double2*>(&rows[j][2 * (threadIdx.x % (D / 2))]);
    if (isfinite(x.x) && isfinite(x.y)) return;
    x = make_double2(isfinite(x.x) ? x.x : 0.0, isfinite(x.y) ? x.y : 0.0);
    atomicOr(bad, bit0 << b);
}
// What spoils two columns, to which v points, of the block's r-th row, which sees keys from first_key on: NaN if it sees a key
// taken out, or a value taken out there; zero otherwise.
template <typename TIn>
__device__ __noinline__ double2 spoilt(const unsigned* bad, Ends ends, int r, int first_key, const TIn* v, long long stride) {
    const unsigned seen = ends.seen(r, first_key);
    double2 x = make_double2(0.0, 0.0);
    if (bad[0] & seen) x = make_double2(NAN, NAN);
    for (int bit = 0; bit < 16; ++bit) {
        if (!(bad[1] & seen & (1u << bit))) continue;
        double a, b;
        load_pair(v + (size_t)(bit < 8 ? ends.hi0 + bit : ends.lo0 + bit - 8) * stride, a, b);
        if (!isfinite(a)) x.x = NAN;
        if (!isfinite(b)) x.y = NAN;
    }
    return x;
}

// out(r)[j] = row(r) . keys[j], eight keys per step of a warp; row and out: pointers of the block's r-th row
template <int D, typename Row, typename Out>
__device__ __forceinline__ void dots(Out&& out, Row&& row, const double (*keys)[DrCfg<D>::LDK], int nkeys, int warp, int lane) {
    using C = DrCfg<D>;
    const int n = lane >> 2, t4 = lane & 3;
    const double* rp = row(n < C::TEAMS ? n : 0);
    for (int kb = warp; 8 * kb < nkeys; kb += C::WARPS) {
        double c[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
        for (int s = 0; s < D / 4; ++s) {
            const double a = rp[4 * s + t4];
            team::dmma(c[s & 1][0], c[s & 1][1], n < C::TEAMS ? a : 0.0, keys[8 * kb + n][4 * s + t4]);
        }
        if (n < C::TEAMS) *reinterpret_cast<double2*>(out(n) + 8 * kb + 2 * t4) = make_double2(c[0][0] + c[1][0], c[0][1] + c[1][1]);
    }
}

}  // namespace lla

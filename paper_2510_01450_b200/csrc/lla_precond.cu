// Preconditioner for the conjugate-gradient solve of the tensor-core forward kernel (Algorithm 2 with a
// preconditioner; the paper runs plain CG).
//
// The system of query row i is C_i = sum_j p_ij (k_j - kbar_i)(k_j - kbar_i)^T + ridge_i I with weights
// p_ij = w_ij / omega_i over the visible keys.  With all weights equal it is the covariance of those keys,
// which is the same matrix for every row that sees the same keys and changes slowly from row to row.  Its
// inverse, formed once per group of key blocks, is a good preconditioner wherever the weights are not far from uniform: on
// the synthetic workloads it takes away more than half of the iterations.  It never changes the solution, only the path to
// it, so it is built in fp32 and stored in fp16; a block whose inversion breaks down gets the identity.
//
// Without a window the rows of a tile see between none and all of the tile's own keys, so those enter with the mean of that, half
// their weight: a row's own covariance is then off by half a block's worth of keys at most, whichever row of the tile it is, and by
// half a group of two blocks past 2048 keys, where two tiles share a matrix.
// (With full weight the first row is off by a whole block: 15.8 instead of 12.1 iterations in the second tile at d = 64, 6.0
// instead of 5.0 in the sixth, three instead of two past 14 K keys at d = 128.)  A chunk of queries whose tiles do not start at a
// block of keys takes the matrix of the block that its tile's last row sees last.
//
// A sliding window moves with the row, so there every query tile has a matrix of its own (two share one where they see 2048 keys
// and more), in which each block of keys has the weight of its mean share in the windows of the tile's rows: the block that the
// first rows see none of, and the one that the last rows have left behind, count by the keys that a row of the tile sees of
// them on average.  The weights lie between zero and one and add up to the mean number of visible keys, which is at least one:
// nothing here divides by zero.
//
// Three kernels, all on the caller's stream ahead of the forward kernel:
//   precond_gram_kernel     a chunk of key blocks each: running sums of k_j k_j^T and k_j inside the chunk, one record per
//                           block that is asked for.  It reads every key once, so it also makes the fp16 copy of k and
//                           finds the largest magnitudes of k and q.  The products run on mma.sync, whose operands come
//                           straight from the tiles (ldmatrix.trans).  16 heads, n = 16384, d = 128: 81 us, twice what
//                           its 280 MB take at the copy bandwidth: eight warps an SM (165 registers a thread) hide a
//                           part of the loads' latency, the top stall.  (Gram sums on the CUDA cores, their scan over
//                           every block and a copy kernel took 430 us)
//   precond_scan_kernel     the sums of whole chunks (the records of their last blocks) become running sums over the sequence
//   precond_invert_kernel   M_g = (G / L - s s^T / L^2 + ridge I)^{-1} with ridge = lambda / L or more, G and s from the records
//                           of the block and of the chunk before it, by Gauss-Jordan elimination in registers, scaled to a largest entry of one
//                           (conjugate gradients do not see the scale of a preconditioner), rounded to fp16.
#include <cuda_fp16.h>

#include <algorithm>

#include "lla_sm100.cuh"

namespace lla {
namespace {

using sm100::max_abs_bf16x2;
using sm100::pack_f16;
using sm100::publish_max_bf16;
using sm100::smem_u32;

constexpr int PC_THREADS = 256;
constexpr int PC_BLOCK = 128;      // keys per Gram block
constexpr int PC_CHUNKS = 32;      // at most
constexpr int PC_QLOADS = 8;       // 16-byte loads in flight of a thread that looks at q

struct PcParams {
    const __nv_bfloat16* k;
    const __nv_bfloat16* q;
    float* gram;       // [units][blocks][D * D + D]
    uint4* k16;        // [units][n][D] fp16
    uint32_t* range;   // the largest magnitudes of k and q (bf16 bit patterns)
    __half* minv;      // [units][blocks][D][D]; with a window the first [tiles] of a unit's are in use
    int n, nb, cb;     // keys; blocks; blocks per chunk
    int chunks, k_blocks;   // chunks of a unit; thread blocks that read k
    int g0;            // first block that a query sees last; with a window the first query tile that is not solved directly
    int tiles;         // query tiles of 128 rows per head
    int B, Hk, H, nq;
    int causal, window, head_rows;
    float lambda;
    Strides sk, sq;
};

__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int D>
__global__ void __launch_bounds__(PC_THREADS)
precond_gram_kernel(const PcParams p) {
    constexpr int LD = D + 8;                       // rows 16 bytes apart modulo 128: ldmatrix without bank conflicts
    constexpr int CPR = D / 8, RPI = PC_THREADS / CPR, NLD = PC_BLOCK / RPI;      // 16-byte pieces per row, rows per step, steps
    constexpr int MT = D / 64, NT = D / 16;         // a warp's tiles of 16 x 8: 4 x 2 warps
    extern __shared__ __align__(16) uint8_t pc_raw[];
    __nv_bfloat16* ks = reinterpret_cast<__nv_bfloat16*>(pc_raw);                     // [2][PC_BLOCK][LD]
    float* sums = reinterpret_cast<float*>(pc_raw + 2 * PC_BLOCK * LD * 2);           // [PC_THREADS][9]
    __shared__ uint32_t s_max[PC_THREADS / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int col = tid % CPR, row0 = tid / CPR;
    // The blocks behind those of k look at q, a tile of one head's rows at a time, whatever its strides.  (Shared out over the blocks
    // of k instead, one load in flight a thread unless q was one piece, 32 heads over one with q as [B, n, H, d] took
    // 0.6 ms longer at n = 4096, d = 128.)
    if ((int)blockIdx.x >= p.k_blocks) {
        constexpr int ROWS = PC_QLOADS * RPI;
        const int tiles = (p.nq + ROWS - 1) / ROWS, all = p.B * p.H * tiles;
        uint32_t q_max = 0;
        for (int t = blockIdx.x - p.k_blocks; t < all; t += gridDim.x - p.k_blocks) {
            const int head = t / tiles, r0 = (t - head * tiles) * ROWS + row0;
            const __nv_bfloat16* src = p.q + p.sq.at(head / p.H, head % p.H, r0) + 8 * col;
            uint4 x[PC_QLOADS];
#pragma unroll
            for (int i = 0; i < PC_QLOADS; ++i)
                x[i] = r0 + i * RPI < p.nq ? *reinterpret_cast<const uint4*>(src + (long long)(i * RPI) * p.sq.r) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int i = 0; i < PC_QLOADS; ++i)
                q_max = max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(max_abs_bf16x2(q_max, x[i].x), x[i].y), x[i].z), x[i].w);
        }
        publish_max_bf16(q_max, p.range + 1, s_max);
        return;
    }
    const int u = blockIdx.x / p.chunks, b0 = (blockIdx.x - u * p.chunks) * p.cb, b1 = min(p.nb, b0 + p.cb);
    const __nv_bfloat16* src = p.k + p.sk.at(u / p.Hk, u % p.Hk, 0) + 8 * col;
    uint4* dst16 = p.k16 + (size_t)u * p.n * CPR + col;
    uint4 raw[NLD];
    auto fetch = [&](int b) {
#pragma unroll
        for (int i = 0; i < NLD; ++i) {
            const int j = b * PC_BLOCK + row0 + i * RPI;
            raw[i] = j < p.n ? *reinterpret_cast<const uint4*>(src + (long long)j * p.sk.r) : make_uint4(0, 0, 0, 0);
        }
    };
    uint32_t k_max = 0;
    float s8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float acc[MT][NT][4] = {};
    const int m0 = (warp & 3) * 16 * MT, n0 = (warp >> 2) * 8 * NT;
    const int mat = lane >> 3, l8 = lane & 7;
    if (b0 < b1) fetch(b0);
    for (int b = b0; b < b1; ++b) {
        __nv_bfloat16* t = ks + (b & 1) * PC_BLOCK * LD;
#pragma unroll
        for (int i = 0; i < NLD; ++i) {
            const int r = row0 + i * RPI, j = b * PC_BLOCK + r;
            *reinterpret_cast<uint4*>(t + r * LD + 8 * col) = raw[i];
            const uint32_t w[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
            uint32_t h[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float x0 = __uint_as_float(w[e] << 16), x1 = __uint_as_float(w[e] & 0xFFFF0000u);
                k_max = max_abs_bf16x2(k_max, w[e]);
                h[e] = pack_f16(x0, x1);
                s8[2 * e] += x0;
                s8[2 * e + 1] += x1;
            }
            if (j < p.n) dst16[(size_t)j * CPR] = make_uint4(h[0], h[1], h[2], h[3]);
        }
        if (b + 1 < b1) fetch(b + 1);
        __syncthreads();
        const uint32_t tb = smem_u32(t);
#pragma unroll 2
        for (int k0 = 0; k0 < PC_BLOCK; k0 += 16) {
            uint32_t a[MT][4], bb[NT / 2][4];      // bb: two tiles of 8 columns each
#pragma unroll
            for (int i = 0; i < MT; ++i)
                ldmatrix_x4_trans(a[i], tb + 2u * ((k0 + (mat >> 1) * 8 + l8) * LD + m0 + 16 * i + (mat & 1) * 8));
#pragma unroll
            for (int i = 0; i < NT / 2; ++i)
                ldmatrix_x4_trans(bb[i], tb + 2u * ((k0 + (mat & 1) * 8 + l8) * LD + n0 + 16 * i + (mat >> 1) * 8));
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int jn = 0; jn < NT; ++jn) mma_bf16(acc[i][jn], a[i], bb[jn >> 1][2 * (jn & 1)], bb[jn >> 1][2 * (jn & 1) + 1]);
        }
        if (p.window > 0 || b == b1 - 1 || precond_block_used(b, p.nb) == b) {
            float* rec = p.gram + ((size_t)u * p.nb + b) * (D * D + D);
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int jn = 0; jn < NT; ++jn) {
                    float* o = rec + (m0 + 16 * i + (lane >> 2)) * D + n0 + 8 * jn + 2 * (lane & 3);
                    *reinterpret_cast<float2*>(o) = make_float2(acc[i][jn][0], acc[i][jn][1]);
                    *reinterpret_cast<float2*>(o + 8 * D) = make_float2(acc[i][jn][2], acc[i][jn][3]);
                }
#pragma unroll
            for (int e = 0; e < 8; ++e) sums[tid * 9 + e] = s8[e];
            __syncthreads();
            if (tid < D) {
                float s = 0.f;
                for (int r = 0; r < RPI; ++r) s += sums[(r * CPR + tid / 8) * 9 + tid % 8];
                rec[D * D + tid] = s;
            }
            __syncthreads();
        }
        // (the next tile goes to the other buffer; the one after it is written behind the next barrier)
    }
    publish_max_bf16(k_max, p.range, s_max);
}

// Records of the chunks' last blocks: running sums over the chunks, element by element (rec: floats of a record).
__global__ void __launch_bounds__(PC_THREADS)
precond_scan_kernel(float* __restrict__ gram, int nb, int cb, int rec) {
    cudaGridDependencySynchronize();
    const int e = blockIdx.x * PC_THREADS + threadIdx.x, chunks = (nb + cb - 1) / cb;
    if (4 * e >= rec) return;
    constexpr int AHEAD = 8;
    float4* p = reinterpret_cast<float4*>(gram + (size_t)blockIdx.y * nb * rec) + e;
    auto at = [&](int c) { return (size_t)(min(nb, (c + 1) * cb) - 1) * (rec / 4); };
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < chunks; c0 += AHEAD) {
        float4 x[AHEAD];
#pragma unroll
        for (int c = 0; c < AHEAD; ++c)
            if (c0 + c < chunks) x[c] = p[at(c0 + c)];
#pragma unroll
        for (int c = 0; c < AHEAD; ++c)
            if (c0 + c < chunks) {
                sum.x += x[c].x; sum.y += x[c].y; sum.z += x[c].z; sum.w += x[c].w;
                if (c0 + c > 0) p[at(c0 + c)] = sum;
            }
    }
}

// The integers t <= y of min(max(t, 0), len) added up.
__device__ __forceinline__ long long sum_clamped(long long y, long long len) {
    return y <= 0 ? 0 : y <= len ? y * (y + 1) / 2 : len * (len + 1) / 2 + (y - len) * len;
}

// The matrix of query tile t under a sliding window: the mean share of key block b in the windows of the tile's rows, which sit
// at the positions first .. last.  (A row at i sees the keys i + 1 - window .. i from zero on.)
__device__ __forceinline__ float window_share(int first, int last, int window, int b, int n) {
    if (b < 0 || PC_BLOCK * b > last) return 0.f;
    const long long len = min(n - PC_BLOCK * b, PC_BLOCK), e = last + 1ll - PC_BLOCK * b, f = first - (long long)PC_BLOCK * b;
    const long long seen = sum_clamped(e, len) - sum_clamped(f, len);
    const long long left = sum_clamped(e - window, len) - sum_clamped(f - window, len);
    return (float)(seen - left) / (float)(len * (last - first + 1));
}

// The sums over keys that a matrix is made of, as records and their weights: what the records of blocks and of chunks before
// them add up to.
constexpr int PC_TERMS = 12;
struct PcTerms {
    int at[PC_TERMS];
    float wt[PC_TERMS];
    int count;
    float keys;      // the weights of all keys
    // the sums up to block b: its own record, and unless it is the last of its chunk that of the chunk before
    __device__ __forceinline__ void sum_to(int b, float weight, int cb, int nb) {
        if (b < 0 || weight == 0.f) return;
        add(b, weight);
        const int before = b / cb * cb - 1;
        if (before >= 0 && b != before + cb && b != nb - 1) add(before, weight);
    }
    __device__ __forceinline__ void add(int record, float weight) {
        for (int i = 0; i < count; ++i)
            if (at[i] == record) { wt[i] += weight; return; }
        at[count] = record;
        wt[count++] = weight;
    }
};

// With a sliding window: every block of keys with its mean share in the windows of the rows of tile g (of two tiles that share).
// (Not inlined: in the kernel's instruction stream it cost the calls without a window 4 us of 237, one head, n = 4096, d = 64.)
__device__ __noinline__ void window_terms(PcTerms* t, int g, int off, int n, int nb, int cb, int window, int head_rows) {
    const bool paired = precond_tiles_paired(g, off, window);
    const int last = min(n - 1, off + PC_BLOCK * g + PC_BLOCK - 1);
    const int first = min(max(off + PC_BLOCK * (paired ? g & ~1 : g), head_rows - 1), last);
    const int hi = last / PC_BLOCK;
    // the shares change at the two blocks that hold the rows (three for two tiles) ...
    const int lo = max(0, first + 1 - window) / PC_BLOCK;
    int lead = max(lo + 2, hi - 2);
    if (paired) {
        // (wide windows: the first keys cut at the nearest block to their mean, at most half a block of sixteen and more.  With the
        // shares of those blocks too an inversion reads up to 14 records: 2300 instead of 2260 us at n = 16384, 8 heads, d = 128,
        // window 2500)
        const int b0 = (max(0, (first + last) / 2 + 1 - window) + PC_BLOCK / 2) / PC_BLOCK;
        t->keys = 0.5f * (float)(first + last) + 1.f - (float)(PC_BLOCK * b0);
        t->sum_to(b0 - 1, -1.f, cb, nb);
        lead = hi - 3;
        window = n;
    } else {
        // ... and at the two that hold the first rows' to the last rows' first keys
        t->keys = (float)(sum_clamped(last + 1, window) - sum_clamped(first, window)) / (float)(last - first + 1);
        for (int b = lo - 1; b <= min(lo + 1, hi); ++b)
            t->sum_to(b, window_share(first, last, window, b, n) - window_share(first, last, window, b + 1, n), cb, nb);
    }
    for (int b = lead; b <= hi; ++b)
        t->sum_to(b, window_share(first, last, window, b, n) - window_share(first, last, window, b + 1, n), cb, nb);
}

// One preconditioner per group of key blocks that tiles ask for (precond_block_used names the group's last block g): the keys
// before the group, those of the group with the mean weight that the group's rows give them.  With a sliding window one per
// query tile or two.
template <int D>
__global__ void __launch_bounds__(PC_THREADS)
precond_invert_kernel(const PcParams p) {
    constexpr int TR = D / 16, V = D / 64;
    constexpr int rec = D * D + D;
    __shared__ float s_red[PC_THREADS / 32];
    __shared__ int s_bad;
    __shared__ PcTerms s_terms;
    __shared__ __align__(16) float s_row[2][D], s_col[2][D];
    __shared__ float sv[D];
    const int u = blockIdx.y, tid = threadIdx.x;
    const int g = p.causal ? p.g0 + (int)blockIdx.x : p.nb - 1;      // the matrix's place; a query tile with a window
    if (p.window > 0) {
        if (g >= p.tiles) return;
        if (precond_tiles_paired(g, p.n - p.nq, p.window) && !(g & 1) && g + 1 < p.tiles) return;      // the odd tile's serves both
        if (tid == 0) {
            s_terms.count = 0;
            window_terms(&s_terms, g, p.n - p.nq, p.n, p.nb, p.cb, p.window, p.head_rows);
        }
    } else {
        if (p.causal && precond_block_used(g, p.nb) != g) return;        // no tile asks for this block's matrix
        if (tid == 0) {
            const int start = precond_group_start(g), hi = min(p.n, PC_BLOCK * (g + 1));
            const float len = (float)(hi - PC_BLOCK * start);
            const float first = (float)max(p.head_rows - PC_BLOCK * start, 0);
            const float w = p.causal ? fminf(fmaxf(0.5f * (first + len) / len, 0.5f), 1.f) : 1.f;
            // (the records are those of blocks g and start - 1 and of the chunks before them, mostly one)
            const int e = start - 1, cg = g / p.cb * p.cb - 1, ce = e < 0 ? -1 : e / p.cb * p.cb - 1;
            const bool more_g = cg >= 0 && g != cg + p.cb && g != p.nb - 1, more_e = ce >= 0 && e != ce + p.cb;
            s_terms.at[0] = g;           s_terms.wt[0] = w;
            s_terms.at[1] = max(e, 0);   s_terms.wt[1] = e < 0 ? 0.f : 1.f - w;
            s_terms.at[2] = max(cg, 0);  s_terms.wt[2] = (more_g ? w : 0.f) + (more_e && ce == cg ? 1.f - w : 0.f);
            s_terms.at[3] = max(ce, 0);  s_terms.wt[3] = more_e && ce != cg ? 1.f - w : 0.f;
            s_terms.count = 4;
            s_terms.keys = (float)(PC_BLOCK * start) + w * len;
        }
    }
    const float* base = p.gram + (size_t)u * p.nb * rec;
    if (tid == 0) s_bad = 0;
    // Thread (ty, tx) of the 16 x 16 grid keeps the entries (64 i + 4 ty + .., 64 j + 4 tx + ..) in registers.
    const int ty = tid >> 4, tx = tid & 15;
    float a[TR][TR] = {};
    float mine = 0.f;
    __syncthreads();
    const float invL = 1.f / s_terms.keys;
    const int terms = s_terms.count;
    cudaGridDependencySynchronize();
    for (int c = 0; c < terms; ++c) {
        const float wt = s_terms.wt[c];
        if (wt == 0.f) continue;
        const float* r = base + (size_t)s_terms.at[c] * rec;
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const float4 x = *reinterpret_cast<const float4*>(r + (64 * (i >> 2) + 4 * ty + (i & 3)) * D + 64 * j + 4 * tx);
                a[i][4 * j] = fmaf(wt, x.x, a[i][4 * j]);
                a[i][4 * j + 1] = fmaf(wt, x.y, a[i][4 * j + 1]);
                a[i][4 * j + 2] = fmaf(wt, x.z, a[i][4 * j + 2]);
                a[i][4 * j + 3] = fmaf(wt, x.w, a[i][4 * j + 3]);
            }
        if (tid < D) mine = fmaf(wt, r[D * D + tid], mine);
    }
    if (tid < D) sv[tid] = mine * invL;
    __syncthreads();
    float sq_part = 0.f;
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < TR; ++j) {
            a[i][j] = fmaf(a[i][j], invL, -sv[64 * (i >> 2) + 4 * ty + (i & 3)] * sv[64 * (j >> 2) + 4 * tx + (j & 3)]);
            sq_part = fmaf(a[i][j], a[i][j], sq_part);
        }
    // Ridge: lambda / L, but at least a 4000th of the covariance's Frobenius norm, which bounds its largest eigenvalue.  The fp16
    // entries of the inverse, the largest of which is one, are off by 2^-12, the matrix as a whole by about 1e-4; without the
    // bound the inverse of keys in a subspace is all ridge, and what it says of the subspace lies below that: r . M r has any sign, and
    // rows with such a matrix needed more iterations than without (keys of rank 60, d = 64, n = 2500: 20.6 instead of
    // 14.6 with 1269 rows at the cap).  Where the spectrum spans more than the bound the iterations grow with the square root of what
    // is beyond (standard deviations from 1 to 0.01: 5 -> 10 iterations, plain conjugate gradients: 64 and more).
    for (int off = 16; off > 0; off >>= 1) sq_part += __shfl_xor_sync(0xffffffffu, sq_part, off);
    if ((tid & 31) == 0) s_red[tid >> 5] = sq_part;
    __syncthreads();
    float sq = 0.f;
    for (int k = 0; k < PC_THREADS / 32; ++k) sq += s_red[k];
    const float ridge = fmaxf(p.lambda * invL, sqrtf(sq) * (1.f / 4000.f));
    if (ty == tx) {
#pragma unroll
        for (int i = 0; i < TR; ++i) a[i][i] += ridge;
    }
    // In-place Gauss-Jordan inversion (no pivoting: the matrix is symmetric positive definite).  Per step the pivot row and
    // the pivot column go through shared memory (two buffers in turn: one barrier per step).  The loops run over the
    // owner of the pivot, so that its place in the owner's registers is a constant (found by comparison instead, 704
    // matrices of 128 x 128 took 430 us; 1150 of them now take 216 us, 256 of 64 x 64 13 us instead of 38).
    bool broke = false;
#pragma unroll
    for (int kh = 0; kh < V; ++kh) {
#pragma unroll 1
        for (int t = 0; t < 16; ++t) {
#pragma unroll
            for (int kl = 0; kl < 4; ++kl) {
                const int ki = 4 * kh + kl, bsel = kl & 1, kk = 64 * kh + 4 * t + kl;
                if (ty == t) {
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        *reinterpret_cast<float4*>(&s_row[bsel][64 * j + 4 * tx]) = make_float4(a[ki][4 * j], a[ki][4 * j + 1], a[ki][4 * j + 2], a[ki][4 * j + 3]);
                }
                if (tx == t) {
#pragma unroll
                    for (int i = 0; i < V; ++i)
                        *reinterpret_cast<float4*>(&s_col[bsel][64 * i + 4 * ty]) = make_float4(a[4 * i][ki], a[4 * i + 1][ki], a[4 * i + 2][ki], a[4 * i + 3][ki]);
                }
                __syncthreads();
                const float piv = s_row[bsel][kk];
                broke |= !(piv > 0.f && piv <= 3e38f);
                const float ip = __fdividef(1.f, piv);
                float rw[TR], cl[TR];
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const float4 x = *reinterpret_cast<const float4*>(&s_row[bsel][64 * j + 4 * tx]);
                    rw[4 * j] = x.x * ip; rw[4 * j + 1] = x.y * ip; rw[4 * j + 2] = x.z * ip; rw[4 * j + 3] = x.w * ip;
                    const float4 y = *reinterpret_cast<const float4*>(&s_col[bsel][64 * j + 4 * ty]);
                    cl[4 * j] = -y.x; cl[4 * j + 1] = -y.y; cl[4 * j + 2] = -y.z; cl[4 * j + 3] = -y.w;
                }
                // every entry as an ordinary one, then the owners of the pivot row and column put theirs right
#pragma unroll
                for (int i = 0; i < TR; ++i)
#pragma unroll
                    for (int j = 0; j < TR; ++j) a[i][j] = fmaf(cl[i], rw[j], a[i][j]);
                if (ty == t) {
#pragma unroll
                    for (int j = 0; j < TR; ++j) a[ki][j] = rw[j];
                }
                if (tx == t) {
#pragma unroll
                    for (int i = 0; i < TR; ++i) a[i][ki] = cl[i] * ip;
                    if (ty == t) a[ki][ki] = ip;
                }
            }
        }
    }
    // the largest entry; store as fp16 scaled to a largest entry of one
    float mx = 0.f;
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < TR; ++j) {
            broke |= !isfinite(a[i][j]);
            mx = fmaxf(mx, fabsf(a[i][j]));
        }
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (broke) s_bad = 1;
    __syncthreads();       // (the sums of the squares have been read)
    if ((tid & 31) == 0) s_red[tid >> 5] = mx;
    __syncthreads();
    mx = 0.f;
    for (int k = 0; k < PC_THREADS / 32; ++k) mx = fmaxf(mx, s_red[k]);
    const bool use_identity = s_bad != 0 || !(mx > 0.f);
    const float sc = use_identity ? 0.f : 1.f / mx;
    __half* dst = p.minv + ((size_t)u * p.nb + g) * D * D;
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const int r = 64 * (i >> 2) + 4 * ty + (i & 3), c = 64 * j + 4 * tx;
            float x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = use_identity ? (r == c + e ? 1.f : 0.f) : a[i][4 * j + e] * sc;
            *reinterpret_cast<uint2*>(dst + r * D + c) = make_uint2(pack_f16(x[0], x[1]), pack_f16(x[2], x[3]));
        }
}

template <int D>
int launch_t(const PcParams& p, int sms, cudaStream_t st) {
    const int units = p.B * p.Hk;
    const size_t smem = 2 * (size_t)PC_BLOCK * (D + 8) * 2 + sizeof(float) * PC_THREADS * 9;
    LLA_CUDA_TRY(cudaFuncSetAttribute(precond_gram_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int rows = PC_QLOADS * (PC_THREADS / (D / 8));
    const long long q_tiles = (long long)p.B * p.H * ((p.nq + rows - 1) / rows);
    precond_gram_kernel<D><<<p.k_blocks + (int)std::min<long long>(q_tiles, 4 * sms), PC_THREADS, smem, st>>>(p);
    LLA_CUDA_TRY(cudaGetLastError());
    // (the two small kernels are programmatic dependents: their launches overlap the kernel before)
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(PC_THREADS);
    cfg.stream = st;
    constexpr int rec = D * D + D;
    if (p.nb > p.cb) {
        cfg.gridDim = dim3((rec / 4 + PC_THREADS - 1) / PC_THREADS, units);
        LLA_CUDA_TRY(cudaLaunchKernelEx(&cfg, precond_scan_kernel, p.gram, p.nb, p.cb, rec));
    }
    cfg.gridDim = dim3(p.window > 0 ? std::max(p.tiles - p.g0, 1) : p.causal ? p.nb - p.g0 : 1, units);
    LLA_CUDA_TRY(cudaLaunchKernelEx(&cfg, precond_invert_kernel<D>, p));
    return LLA_OK;
}

}  // namespace

int precond_blocks(int n) { return (n + PC_BLOCK - 1) / PC_BLOCK; }

size_t precond_gram_bytes(int units, int n, int d) {
    return ((size_t)units * precond_blocks(n) * ((size_t)d * d + d) * sizeof(float) + 255) & ~(size_t)255;
}
size_t precond_minv_bytes(int units, int n, int d) {
    return ((size_t)units * precond_blocks(n) * (size_t)d * d * sizeof(__half) + 255) & ~(size_t)255;
}

int launch_precond(const ForwardArgs& a, void* k16, uint32_t* range, void* gram, void* minv) {
    PcParams p = {};
    p.k = static_cast<const __nv_bfloat16*>(a.k); p.q = static_cast<const __nv_bfloat16*>(a.q);
    p.gram = static_cast<float*>(gram); p.k16 = static_cast<uint4*>(k16); p.range = range; p.minv = static_cast<__half*>(minv);
    p.n = a.n; p.nb = precond_blocks(a.n);
    p.B = a.B; p.Hk = a.H / a.kv_group; p.H = a.H; p.nq = a.nq;
    int dev = 0, sms = 0;
    LLA_CUDA_TRY(cudaGetDevice(&dev));
    LLA_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // chunks: two thread blocks an SM at d = 64 and one at d = 128, where the registers hold no more, whatever the number of heads
    // (with eight chunks always, one key/value head had eight blocks in all: 32 heads over one, n = 4096, d = 128: 70 us more).
    // Many heads keep eight: with 16 chunks 16 heads of 16384 keys took 83 us instead of 78.
    const int units = p.B * p.Hk;
    const int most = std::min(std::max((a.d == 64 ? 2 : 1) * sms / units, 8), PC_CHUNKS);
    p.cb = (p.nb + most - 1) / most;
    if (p.cb > 1) p.cb += p.cb & 1;      // a chunk's last block is then one whose record is written anyway
    p.chunks = (p.nb + p.cb - 1) / p.cb;
    p.k_blocks = p.chunks * units;
    p.causal = a.causal; p.window = a.causal ? a.window : 0; p.head_rows = a.head_rows > 0 ? a.head_rows : 0;
    p.tiles = (a.nq + PC_BLOCK - 1) / PC_BLOCK;
    p.g0 = p.window > 0 ? head_rows_count(a) / PC_BLOCK          // (rows before are solved directly)
                        : std::max(a.n - a.nq, std::min(a.n, p.head_rows) - 1) / PC_BLOCK;
    p.lambda = a.lambda; p.sk = a.sk; p.sq = a.sq;
    if (a.d == 64) return launch_t<64>(p, sms, a.stream);
    if (a.d == 128) return launch_t<128>(p, sms, a.stream);
    return LLA_ERR_UNSUPPORTED;
}

}  // namespace lla

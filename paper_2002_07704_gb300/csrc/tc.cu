// Tensor-core form of the truncated block product in split TF32: precision LSQ_TF32X3 (4 x 4 blocks), and
// the LSQ_F32 products that split_choice gives it (also of 9 x 9 to 16 x 16 blocks, as 4 x 4 units).
//
// Sec. 2.3.2 of the paper: every product of the linear-scaling method is restricted to the
// range of its result, C_ij = sum_k A_ik B_kj over the stored blocks (i, j) of C.  Here the
// 4 x 4 blocks are contracted on the tensor cores (tcgen05.mma, kind::tf32, FP32
// accumulation in tensor memory):
//
//  * Split TF32 operands.  Every float32 value v is held as hi = tf32(v) and
//    lo = tf32(v - hi), so hi + lo carries v to 22 bits.  A block is one 128-byte unit: the
//    4 x 4 hi values (row-major), then the 4 x 4 lo values.
//  * Tiles.  Atoms i are taken in groups of 16 (two diamond cells in cell-ordered systems).
//    The atoms j of the group's rows of C are cut into tiles of 32, and each tile has one
//    list of atoms k: the union of the group's rows of op(A), restricted to atoms that the
//    tile's rows of op(B)^T hold (padded to a multiple of 16).  A tile is one accumulator of
//    M = 128 rows (16 i x {hi, lo} x 4 rows r of A_ik) by N = 256 columns (32 j x {hi, lo} x 4
//    rows c of X_jk = (B_kj)^T), and one MMA takes K = 8 (two atoms k x 4).  The {hi, lo} x
//    {hi, lo} cross terms land in separate rows and columns and are summed in the epilogue:
//    one pass gives hi.hi + hi.lo + lo.hi + lo.lo.  Larger tiles copy fewer blocks a triple
//    (SL.Q^T of 4096 atoms: 8 x 16 165 M, 16 x 32 125 M; L.S.L 130 and 89 M) though fewer of
//    their dense triples are stored ones (33 and 20 %): 2644 -> 2236 and 3325 -> 2855 us.
//  * Gathers.  The blocks of a stage (8 k of the list for the 32 rows j and the 16 rows i)
//    are copied into shared memory by 16-byte asynchronous copies (cp.async), eight lanes
//    per 128-byte block, so one warp instruction moves four whole cache lines; for a block
//    that a row does not hold the copy writes zeros and reads nothing.  The block indices a
//    CTA gathers are laid out by the plan as one stream of stage records, itself copied to
//    shared memory eight stages ahead, so no copy waits on an index load.  The kernel is
//    bound by shared memory, which the copies write (48 KB a stage, 384 cycles) and the MMAs
//    read (12 KB each, 384 cycles a stage), and by the rate of the gathers (about 10 TB/s of
//    scattered 128-byte lines), not by DRAM.  (Bulk copies of runs of consecutive blocks were
//    measured first: at the ~4 blocks a run averages, their request rate, not the bytes,
//    bounded the kernel.)
//    (With every block absent, one MMA a stage and no sums, issuing the 96 copy instructions
//    of a stage still takes 700 cycles of the 1200 to 1250 measured at 1728 atoms.)
//  * Roles.  Six warps issue the copies through a ring of stages, one thread issues the
//    MMAs, sixteen warps read the accumulator (tcgen05.ld) and write the blocks of C the plan
//    keeps.  The tensor core's float32 additions truncate, which biases long sums, so every
//    two stages (8 MMAs) fill a fresh accumulator, of two in tensor memory, and the epilogue
//    adds these in float32 with rounding to nearest (every stage for LSQ_F32).  Every wait on an mbarrier is bounded:
//    past the limit the kernel records an error code in a device word, stops issuing work,
//    waits (bounded) for its copies and MMAs in flight, frees its tensor memory and returns.
//
// The plan (which blocks to gather, where to write) is built on the GPU once per geometry
// and product, like the FMA path's plan.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <functional>
#include <queue>
#include <string>
#include <utility>
#include <vector>

#include "listed.h"
#include "lsq_internal.h"
#include "tc_ptx.h"

namespace lsq {
namespace {

// Tiles of this kernel (in sub-rows for larger blocks, see TcTile): 16 atoms i by 32 atoms j, 8 atoms k
// a stage.
constexpr int kGI = 16, kJ = 32;
constexpr int kRowsT = kJ + kGI;              // gathered rows per stage
constexpr int kKT = 8;                        // atoms k per stage
constexpr int kStages = 4;                    // stages in the ring
constexpr int kUnit = 128;                    // bytes of a split block (hi 64, lo 64)
constexpr int kPanelX = kJ * kKT * kUnit;     // X rows of a stage (N side), 32 KB
constexpr int kStageBytes = kRowsT * kKT * kUnit;  // 48 KB
constexpr int kBufCols = 8 * kJ;              // accumulator columns
constexpr int kBufs = 2;                      // accumulators in tensor memory
constexpr int kTmemCols = kBufs * kBufCols;   // all 512
constexpr int kCopyWarps = 6;                 // warps 0-5 copy (8 rows of a stage each)
constexpr int kMmaWarp = 6;                   // one thread of warp 6 issues the MMAs
constexpr int kEpiWarp = 7, kEpiWarps = 16;   // warps 7-22 read the accumulators
constexpr int kThreads = 32 * (kEpiWarp + kEpiWarps);
constexpr int kRecT = kRowsT * kKT;           // entries of a stage record
constexpr int kRecRing = 16, kRecAhead = 8;   // records in shared memory
constexpr int kRingBytes = kRecRing * kRecT * 4;
constexpr uint16_t kAbsent = 0xffff;

__device__ __forceinline__ bool tri_skip_tc(int tri, int i, int j) {
    return tri == 1 ? j < i : (tri == 2 ? j > i : false);
}

// ---- split TF32 operands -------------------------------------------------------------
// Round to the nearest tf32 value (10 fraction bits), halfway cases away from zero: add
// half a unit of the 11th bit to the magnitude bits, then clear the 13 low bits.
__device__ __forceinline__ float tf32_round(float v) {
    return __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
}

// Unit (R, K) of block p (rows 4 R .., columns 4 K ..; zeros beyond b): hi and lo of X (MODE 0), of X^T
// read through the transpose map tm (MODE 1; block (i, j) of X^T is (X_ji)^T), or of X + X^T (MODE 2, X
// on a symmetric pattern; the sum rounded once in float32, as a separate symmetric sum would).  v - hi
// is exact in float32.  With range, its words become the largest bits of |v| and of their complement
// over the finite nonzero values, the largest and the smallest (see least_sum), and 1 if a value is not
// finite.  An infinity or NaN gives parts that are NaN, whatever its bits.  any: a byte a unit, 0 if it
// is all zeros.
// A thread takes a row of a unit: one 16-byte load where blocks are 4 x 4, X is aligned (vec) and not
// transposed, two 16-byte stores.  Bound by HBM.
template <int MODE, int NB>
__global__ void __launch_bounds__(256) k_split_tf32(int64_t nnzb, int b, const int64_t *__restrict__ tm,
                                                    const float *__restrict__ X, bool vec, float4 *__restrict__ out,
                                                    unsigned *__restrict__ range, uint8_t *__restrict__ any) {
    const int64_t m = nnzb * (4 * NB * NB);
    unsigned most = 0, least = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = e >> 2, p = u / (NB * NB);
        const int r = (int)(e & 3);
        float v[4];
        if constexpr (NB == 1) {
            if (MODE != 1) {
                if (vec) {
                    const float4 x = __ldg(reinterpret_cast<const float4 *>(X) + e);
                    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[c] = __ldg(X + 4 * e + c);
                }
            }
            if (MODE != 0) {
                const float *T = X + 16 * tm[p] + r;
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] = MODE == 1 ? __ldg(T + 4 * c) : v[c] + __ldg(T + 4 * c);
            }
        } else {
            const int row = 4 * ((int)(u / NB) % NB) + r, col = 4 * (int)(u % NB), bb = b * b;
            const int64_t q = MODE ? tm[p] : p;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                v[c] = 0.f;
                if (row < b && col + c < b) {
                    if (MODE != 1) v[c] = __ldg(X + bb * p + row * b + col + c);
                    if (MODE != 0) v[c] += __ldg(X + bb * q + (col + c) * b + row);
                }
            }
        }
        float hi[4], lo[4];
        bool some = false;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const unsigned m = __float_as_uint(v[c]) & 0x7fffffffu;
            some = some || m != 0;
            if (m >= 0x7f800000u) {
                v[c] = __uint_as_float(0x7fc00000u);
                if (range) range[2] = 1;
            } else if (m != 0) {
                most = max(most, m);
                least = max(least, 0x7fffffffu - m);
            }
            hi[c] = tf32_round(v[c]);
            lo[c] = tf32_round(v[c] - hi[c]);
        }
        if (any) {
            // the unit's four rows are four neighbouring lanes
            const unsigned rows = __ballot_sync(0xfu << (threadIdx.x & 28), some);
            if (r == 0) any[u] = rows != 0;
        }
        out[8 * u + r] = make_float4(hi[0], hi[1], hi[2], hi[3]);
        out[8 * u + 4 + r] = make_float4(lo[0], lo[1], lo[2], lo[3]);
    }
    if (range) {
        __shared__ unsigned sh[2];
        if (threadIdx.x < 2) sh[threadIdx.x] = 0;
        __syncthreads();
        most = __reduce_max_sync(0xffffffffu, most);
        least = __reduce_max_sync(0xffffffffu, least);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(sh, most);
            atomicMax(sh + 1, least);
        }
        __syncthreads();
        // (few thread blocks find the words smaller than theirs)
        if (threadIdx.x < 2 && sh[threadIdx.x] > static_cast<volatile unsigned *>(range)[threadIdx.x])
            atomicMax(range + threadIdx.x, sh[threadIdx.x]);
    }
}

// ---- plan ------------------------------------------------------------------------------
// Number of entries of pos[0, m) that name a block (>= 0).
__global__ void k_count_present(int64_t m, const int32_t *__restrict__ pos, unsigned long long *__restrict__ out) {
    unsigned long long c = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        c += pos[e] >= 0 ? 1ull : 0ull;
    for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

struct TcBuild {
    int n, ngroups, upper;
    TcTile tile;
    __device__ int G() const { return tile.G; }
    __device__ int JT() const { return tile.JT; }
    __device__ int KS() const { return tile.KS; }
    __device__ int rec() const { return (tile.G + tile.JT) * tile.RK; }
    __device__ int rec_at(int r, int k) const {
        if (tile.RK < 8) return r * tile.RK + k;
        return r * 8 + (tile.kind == 0 ? 4 * (k & 1) + (k >> 1) : 2 * (k & 3) + (k >> 2));
    }
    const int64_t *a_ptr, *x_ptr, *c_ptr;
    const int32_t *a_col, *x_col, *c_col;
    const int32_t *g_toff;        // [ngroups + 1] first tile of each group
    int32_t *tile_j;              // [JT ntiles]
    int32_t *tile_nk;             // [ntiles]
    const int64_t *tile_posoff;   // [ntiles]
    const int64_t *tile_koff;     // [ntiles] start of the tile's k-list in klist
    int32_t *klist;               // scratch
    int32_t *pos;
    int32_t *cpos;
};

__device__ __forceinline__ void clear_bits(uint32_t *bm, int W) {
    for (int w = threadIdx.x; w < W; w += blockDim.x) bm[w] = 0u;
}

// bm |= the columns of row r (those within the triangle tri of row r when tri > 0).
__device__ __forceinline__ void or_row(const int64_t *__restrict__ ptr, const int32_t *__restrict__ col, int r,
                                       int tri, uint32_t *bm) {
    for (int64_t q = ptr[r] + threadIdx.x; q < ptr[r + 1]; q += blockDim.x) {
        const int c = col[q];
        if (!tri_skip_tc(tri, r, c)) atomicOr(&bm[c >> 5], 1u << (c & 31));
    }
}

// Sum of v over the block (every thread receives it).  sh: 32 ints of shared memory.
__device__ int block_sum(int v, int *sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    __syncthreads();
    return t;
}

// Exclusive prefix sum of v over the block; *total receives the sum.  sh: 32 ints.
__device__ int block_scan_excl(int v, int *total, int *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < nw ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) sh[lane] = w;
    }
    __syncthreads();
    const int before = (warp > 0 ? sh[warp - 1] : 0) + x - v;
    *total = sh[nw - 1];
    __syncthreads();
    return before;
}

// Writes the set bits of bm[0..W) in ascending order to out[0..); returns their number.
__device__ int compact_bits(const uint32_t *bm, int W, int32_t *out, int *sh) {
    const int chunk = (W + (int)blockDim.x - 1) / (int)blockDim.x;
    const int w0 = min(W, (int)threadIdx.x * chunk), w1 = min(W, w0 + chunk);
    int v = 0;
    for (int w = w0; w < w1; ++w) v += __popc(bm[w]);
    int total;
    int r = block_scan_excl(v, &total, sh);
    for (int w = w0; w < w1; ++w) {
        uint32_t bits = bm[w];
        while (bits) {
            const int b = __ffs(bits) - 1;
            bits &= bits - 1u;
            out[r++] = 32 * w + b;
        }
    }
    return total;
}

// Pass 1: tiles of each group (its atoms j: the union of its rows of C within the triangle).
__global__ void __launch_bounds__(512) k_tc_groups(TcBuild a, int32_t *__restrict__ nt_out) {
    extern __shared__ __align__(16) uint32_t jb[];
    __shared__ int sh[32];
    const int W = (a.n + 31) >> 5;
    for (int g = blockIdx.x; g < a.ngroups; g += gridDim.x) {
        clear_bits(jb, W);
        __syncthreads();
        for (int i = a.G() * g; i < min(a.G() * (g + 1), a.n); ++i) or_row(a.c_ptr, a.c_col, i, a.upper, jb);
        __syncthreads();
        int c = 0;
        for (int w = threadIdx.x; w < W; w += blockDim.x) c += __popc(jb[w]);
        c = block_sum(c, sh);
        if (threadIdx.x == 0) nt_out[g] = (c + a.JT() - 1) / a.JT();
        __syncthreads();
    }
}

// Pass 2: atoms j of each tile and the length of its k-list (a multiple of KS).
__global__ void __launch_bounds__(512) k_tc_tiles(TcBuild a) {
    extern __shared__ __align__(16) uint32_t bm[];
    __shared__ int sh[32];
    const int W = (a.n + 31) >> 5;
    uint32_t *kb = bm, *jb = bm + W, *tb = bm + 2 * W;
    for (int g = blockIdx.x; g < a.ngroups; g += gridDim.x) {
        const int i0 = a.G() * g, i1 = min(i0 + a.G(), a.n);
        clear_bits(kb, 2 * W);
        __syncthreads();
        for (int i = i0; i < i1; ++i) {
            or_row(a.a_ptr, a.a_col, i, 0, kb);
            or_row(a.c_ptr, a.c_col, i, a.upper, jb);
        }
        __syncthreads();
        const int t0 = a.g_toff[g], nt = a.g_toff[g + 1] - t0;
        const int cj = compact_bits(jb, W, a.tile_j + (int64_t)a.JT() * t0, sh);
        for (int m = cj + threadIdx.x; m < a.JT() * nt; m += blockDim.x) a.tile_j[(int64_t)a.JT() * t0 + m] = -1;
        __syncthreads();
        for (int t = t0; t < t0 + nt; ++t) {
            clear_bits(tb, W);
            __syncthreads();
            for (int jj = 0; jj < a.JT(); ++jj) {
                const int j = a.tile_j[(int64_t)a.JT() * t + jj];
                if (j >= 0) or_row(a.x_ptr, a.x_col, j, 0, tb);
            }
            __syncthreads();
            int c = 0;
            for (int w = threadIdx.x; w < W; w += blockDim.x) c += __popc(tb[w] & kb[w]);
            c = block_sum(c, sh);
            if (threadIdx.x == 0) a.tile_nk[t] = max(a.KS(), (c + a.KS() - 1) / a.KS() * a.KS());
            __syncthreads();
        }
    }
}

// map[col] = offset of col in row r (set) or kAbsent (unset), for one row at a time.
__device__ __forceinline__ void map_row(const int64_t *__restrict__ ptr, const int32_t *__restrict__ col, int r,
                                        uint16_t *map, bool set) {
    const int64_t p0 = ptr[r], p1 = ptr[r + 1];
    for (int64_t q = p0 + threadIdx.x; q < p1; q += blockDim.x) map[col[q]] = set ? (uint16_t)(q - p0) : kAbsent;
}

// Pass 3: each tile's k-list, the index of each listed block in the tile's G + JT rows (stage
// records), and the positions in C of the blocks (i, j) the tile writes.
__global__ void __launch_bounds__(512) k_tc_fill(TcBuild a) {
    extern __shared__ __align__(16) uint32_t bm[];
    __shared__ int sh[32];
    const int W = (a.n + 31) >> 5;
    uint32_t *kb = bm, *tb = bm + W;
    uint16_t *map = reinterpret_cast<uint16_t *>(bm + 2 * W);
    for (int e = threadIdx.x; e < a.n; e += blockDim.x) map[e] = kAbsent;
    __syncthreads();
    for (int g = blockIdx.x; g < a.ngroups; g += gridDim.x) {
        const int i0 = a.G() * g, i1 = min(i0 + a.G(), a.n);
        const int t0 = a.g_toff[g], nt = a.g_toff[g + 1] - t0;
        clear_bits(kb, W);
        __syncthreads();
        for (int i = i0; i < i1; ++i) or_row(a.a_ptr, a.a_col, i, 0, kb);
        __syncthreads();
        for (int t = t0; t < t0 + nt; ++t) {
            clear_bits(tb, W);
            __syncthreads();
            for (int jj = 0; jj < a.JT(); ++jj) {
                const int j = a.tile_j[(int64_t)a.JT() * t + jj];
                if (j >= 0) or_row(a.x_ptr, a.x_col, j, 0, tb);
            }
            __syncthreads();
            for (int w = threadIdx.x; w < W; w += blockDim.x) tb[w] &= kb[w];
            __syncthreads();
            const int nk = a.tile_nk[t];
            const int64_t po = a.tile_posoff[t];
            int32_t *kl = a.klist + a.tile_koff[t];
            const int ck = compact_bits(tb, W, kl, sh);
            // The float32 sums take the list from the first atom beyond the tile's, and around to the
            // tile's own: the largest terms, at atoms k near i and j, then come late, after sums that
            // are still small (rounding loses as much as the sum is large).
            int past = 0, last = i1 - 1;
            for (int jj = 0; jj < a.JT(); ++jj) last = max(last, a.tile_j[(int64_t)a.JT() * t + jj]);
            for (int w = threadIdx.x; w < W; w += blockDim.x) {
                const int n0 = last - 32 * w;  // bits 0 .. n0 of the word are atoms up to `last`
                past += n0 < 0 ? 0 : __popc(n0 >= 31 ? tb[w] : tb[w] & ((2u << n0) - 1u));
            }
            past = block_sum(past, sh);
            const int turn = a.tile.kind == 1 && ck > 0 ? past % ck : 0;
            auto k_at = [&](int m) { return m < ck ? kl[m + turn < ck ? m + turn : m + turn - ck] : -1; };
            __syncthreads();
            for (int r = 0; r < a.JT() + a.G(); ++r) {
                int row;
                const int64_t *ptr;
                const int32_t *col;
                if (r < a.JT()) {
                    row = a.tile_j[(int64_t)a.JT() * t + r];
                    ptr = a.x_ptr;
                    col = a.x_col;
                } else {
                    row = i0 + r - a.JT() < a.n ? i0 + r - a.JT() : -1;
                    ptr = a.a_ptr;
                    col = a.a_col;
                }
                const int64_t row0 = row >= 0 ? ptr[row] : 0;
                if (row >= 0) map_row(ptr, col, row, map, true);
                __syncthreads();
                for (int m = threadIdx.x; m < nk; m += blockDim.x) {
                    const int k = k_at(m);
                    const uint16_t o = (row >= 0 && k >= 0) ? map[k] : kAbsent;
                    a.pos[po + (int64_t)a.rec() * (m / a.tile.RK) + a.rec_at(r, m % a.tile.RK)] =
                        o == kAbsent ? -1 : (int32_t)(row0 + o);
                }
                __syncthreads();
                if (row >= 0) map_row(ptr, col, row, map, false);
                __syncthreads();
            }
        }
        for (int rr = 0; rr < a.G(); ++rr) {
            const int i = i0 + rr;
            if (i < i1) map_row(a.c_ptr, a.c_col, i, map, true);
            __syncthreads();
            for (int m = threadIdx.x; m < a.JT() * nt; m += blockDim.x) {
                const int t = t0 + m / a.JT(), jj = m % a.JT();
                const int j = a.tile_j[(int64_t)a.JT() * t0 + m];
                int32_t v = -1;
                if (i < i1 && j >= 0 && !tri_skip_tc(a.upper, i, j) && map[j] != kAbsent)
                    v = (int32_t)(a.c_ptr[i] + map[j]);
                a.cpos[(int64_t)a.G() * a.JT() * t + a.JT() * rr + jj] = v;
            }
            __syncthreads();
            if (i < i1) map_row(a.c_ptr, a.c_col, i, map, false);
            __syncthreads();
        }
    }
}

// Marks the blocks of C of each tile that no stored pair of blocks adds to: entry v of cpos becomes
// -2 - v.  Bits of a row's listed blocks, 1024 atoms k at a time, against those of each other row.
constexpr int kMaxRows = kGI + kJ, kMaxPairs = kGI * kJ;  // of a tile of either kind
__global__ void __launch_bounds__(256) k_tc_empty(TcBuild a, int ntiles) {
    constexpr int kW = 32, kMine = kMaxPairs / 256;
    __shared__ uint32_t bits[kMaxRows][kW + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, R = a.G() + a.JT(), pairs = a.G() * a.JT();
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int nk = a.tile_nk[t];
        const int32_t *pos = a.pos + a.tile_posoff[t];
        uint32_t hit[kMine] = {};
        for (int k0 = 0; k0 < nk; k0 += 32 * kW) {
            for (int e = warp; e < R * kW; e += blockDim.x >> 5) {
                const int r = e / kW, w = e % kW, m = k0 + 32 * w + lane;
                const bool on = m < nk && pos[(int64_t)a.rec() * (m / a.tile.RK) + a.rec_at(r, m % a.tile.RK)] >= 0;
                const uint32_t word = __ballot_sync(0xffffffffu, on);
                if (lane == 0) bits[r][w] = word;
            }
            __syncthreads();
#pragma unroll
            for (int h = 0; h < kMine; ++h) {
                const int q = threadIdx.x + 256 * h;
                if (q < pairs)
                    for (int w = 0; w < kW; ++w) hit[h] |= bits[a.JT() + q / a.JT()][w] & bits[q % a.JT()][w];
            }
            __syncthreads();
        }
#pragma unroll
        for (int h = 0; h < kMine; ++h) {
            const int q = threadIdx.x + 256 * h;
            if (q < pairs && hit[h] == 0) {
                int32_t &v = a.cpos[(int64_t)pairs * t + q];
                if (v >= 0) v = -2 - v;
            }
        }
    }
}

// ---- the product -----------------------------------------------------------------------
struct TcArgs {
    int b;
    int c_vec;  // C is 16-byte aligned
    const int32_t *order, *cta_first, *tile_nk, *cpos, *cta_stages;
    const int64_t *cta_rec;  // first record of each CTA's stream
    const int32_t *pos;
    const char *As, *Xs;  // split units of op(A) and of X = op(B)^T
    float *C;
    const int64_t *c_tm;  // transpose map of C's pattern: also write C_ji = C_ij^T (or null)
    float alpha, beta;
    // LSQ_F32: the smallest and largest values of op(A) and of X (see k_split_tf32), and the units left to
    // k_listed: their number, ((row, sub-row, sub-column), block)
    const unsigned *range;
    int *count;
    int2 *list;
    const int32_t *tile_i0;
    int log_terms;  // 2^log_terms: no sum has more terms
    int *err;
    unsigned long long wait_ns;  // bound of the pipeline waits (the final drain keeps kWaitNs)
};

// NB: 4 x 4 units along a side of a block.  FL: stages to an accumulator.  The tensor core's float32
// additions truncate, which biases long sums, so FL stages (8 FL atoms k) fill a fresh accumulator and
// these are added by the epilogue, rounded to nearest.  FL = 2 for LSQ_TF32X3; FL = 1 for LSQ_F32,
// whose FMA kernels it replaces: 2-norm of the error, SL.Q^T of 4096 atoms, 2.2e-7 (FL = 2), 1.9e-7
// (FL = 1) and 3.8e-7 in FMA; LS.L of 512 atoms 1.9e-7, 1.5e-7 and 1.8e-7.  FL = 1 costs 14 %.
//
// A sum of the split is as good as FMA's (to 2^-25 of itself) down to this size.  The tensor cores may
// flush what lies below 2^-126: products of the parts of small values, and the lo part of values
// below 2^-102 (or all of a subnormal one) times whatever they meet.  Blocks with smaller sums, or
// sums that are no numbers, are listed for k_listed; others are not, whatever their operands hold.
// *zero: sums up to this size are not listed either: 0 if no value and no product of two can be flushed
// as a whole (a sum of 0 then has no terms, or ones that cancel), else -1.  (Structural zeros are many:
// with those of a 13-orbital model listed, and no note of the stored zero units, a batch step took
// 387 ms instead of 220.)
// (One value beyond 2^60 or below 2^-100 used to send the whole product to a kernel like k_listed.
// That takes 5 to 10 times as long as the FMA schedules when it has every block to do, 19.6 ms against
// 3.5 for the products of a gradient of 989 atoms: it has no plan to find pairs with.)
__device__ __forceinline__ float least_sum(const unsigned *range, int log_terms, float *zero) {
    *zero = 0.f;
    if (range[0] == 0 || range[4] == 0) return 0.f;  // an operand without finite nonzero values
    const int ma = (int)(range[0] >> 23) - 126, mx = (int)(range[4] >> 23) - 126;  // below 2^m
    const int la = (int)((0x7fffffffu - range[1]) >> 23) - 127, lx = (int)((0x7fffffffu - range[5]) >> 23) - 127;
    if (la < -126 || lx < -126 || la + lx < -124) *zero = -1.f;
    int lost = -1000;  // log2 of what a term can lose
    if (la + lx - 48 < -126) lost = -126 + 2;
    if (la < -102) lost = max(lost, -126 + max(mx, 0) + 1);
    if (lx < -102) lost = max(lost, -126 + max(ma, 0) + 1);
    const int least = lost + log_terms + 25;
    if (la + lx >= least) return 0.f;  // the smallest product there can be is as large
    return ldexpf(1.f, min(least, 127));
}

template <int NB, int FL>
__global__ void __launch_bounds__(kThreads, 1) k_tc_product(TcArgs p) {
    constexpr int kRecN = kRecT / (NB * NB);  // entries of a record
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kStages * kStageBytes + kRingBytes);
    // bars: full[kStages], empty[kStages], tfull[kBufs], tempty[kBufs], drain[1]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStages + 2 * kBufs + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto empty = [&](int s) { return bar0 + 8u * (kStages + s); };
    auto tfull = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
    auto tempty = [&](int b) { return bar0 + 8u * (2 * kStages + kBufs + b); };
    const uint32_t drain = bar0 + 8u * (2 * kStages + 2 * kBufs);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q0 = p.cta_first[blockIdx.x], q1 = p.cta_first[blockIdx.x + 1];

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full(s), 32 * kCopyWarps);  // per copying thread: its copies have landed
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < kBufs; ++b) {
            mbar_init(tfull(b), 1);
            mbar_init(tempty(b), kEpiWarps);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp < kCopyWarps) {
        // ---- copies.  Warp w fills rows 8w .. 8w + 7 of every stage (rows 0-31: atoms j of the
        // tile, rows of X; 32-47: atoms i of the group, rows of op(A)).  One instruction moves
        // four blocks of a row: lane l copies 16-byte chunk l % 8 of block 4 h + l / 8 (h = 0, 1).
        // The stage records, read from HBM once each, are copied into a ring in shared memory
        // kRecAhead stages ahead (a wait on empty(slot) below means that the copies of four
        // stages back, and the record copies before them, have landed).
        const char *arr = (warp < 4 ? p.Xs : p.As) + 16 * (lane & 7) + (NB == 1 ? 0 : kUnit * (lane >> 3));
        const int S = 2 * p.cta_stages[blockIdx.x], sub = lane >> 3;
        constexpr int kWarpRec = NB == 1 ? 64 : 4;
        const int32_t *rec = p.pos + p.cta_rec[blockIdx.x] + kWarpRec * warp;
        const uint32_t ring = sbase + kStages * kStageBytes + 4 * kWarpRec * warp;
        auto fetch = [&](int st) {
            if (st < S && lane < kWarpRec / 4)
                cp_async16(ring + (uint32_t)(st % kRecRing) * (4 * kRecN) + 16 * lane, rec + (int64_t)kRecN * st + 4 * lane);
        };
        for (int st = 0; st < kRecAhead; ++st) fetch(st);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        const uint32_t dlane = (uint32_t)(8 * warp * kKT * kUnit + sub * kUnit + 16 * (lane & 7));
        for (int st = 0; st < S; ++st) {
            const int slot = st % kStages;
            bool ok = mbar_wait(empty(slot), ((uint32_t)(st / kStages) & 1u) ^ 1u, abort_flag, p.err, 1, p.wait_ns);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const uint32_t dst = sbase + (uint32_t)slot * kStageBytes + dlane;
            const uint32_t from = ring + (uint32_t)(st % kRecRing) * (4 * kRecN);
            fetch(st + kRecAhead);
            if constexpr (NB == 1) {
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    int v[2];
                    asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(from + 32 * r + 8 * sub) : "memory");
#pragma unroll
                    for (int h = 0; h < 2; ++h) cp_async16_or_zero(dst + (r * kKT + 4 * h) * kUnit, arr, v[h], kUnit);
                }
            } else {
                // two atoms of four sub-rows each; the stage's eight k are the sub-columns of two atoms
                int v[4];
                asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(from) : "memory");
#pragma unroll
                for (int r = 0; r < 8; ++r)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        cp_async16_or_zero(dst + (r * kKT + 4 * h) * kUnit, arr + kUnit * NB * (r & 3), v[2 * (r >> 2) + h],
                                           NB * NB * kUnit);
            }
            cp_async_arrive(full(slot));
        }
        // every copy of this thread has landed before the CTA exits
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            // ---- MMAs: per stage 4 of M = 128 (16 i), N = 256 (32 j), K = 8 (two atoms k).  (Two of 16 j by
            // 16 i instead read a third more shared memory, which the copies need too.)
            constexpr uint32_t idesc = idesc_tf32(8 * kGI, kBufCols);
            int it = 0, st = 0;
            bool ok = true;
            int nk_n = q0 < q1 ? __ldg(p.tile_nk + __ldg(p.order + q0)) : 0;
            for (int q = q0; q < q1 && ok; ++q) {
                const int nk = nk_n;
                if (q + 1 < q1) nk_n = __ldg(p.tile_nk + __ldg(p.order + q + 1));
                for (int k0 = 0; k0 < nk && ok; k0 += FL * kKT / NB, ++it) {
                    const int buf = it % kBufs;
                    ok = mbar_wait(tempty(buf), ((uint32_t)(it / kBufs) & 1u) ^ 1u, abort_flag, p.err, 3, p.wait_ns);
                    if (!ok) break;
                    for (int h = 0; h < FL; ++h, ++st) {
                        const int slot = st % kStages;
                        ok = mbar_wait(full(slot), (uint32_t)(st / kStages) & 1u, abort_flag, p.err, 2, p.wait_ns);
                        if (!ok) break;
                        // the stage was written by cp.async (generic proxy); the MMAs read it
                        // through the async proxy
                        fence_proxy_async();
                        tc_fence_after();
                        const uint32_t sx = sbase + (uint32_t)slot * kStageBytes, sa = sx + kPanelX;
#pragma unroll
                        for (int kk = 0; kk < kKT; kk += 2)
                            mma_tf32(tmem + (uint32_t)(buf * kBufCols), sdesc(sa + kk * kUnit, kUnit, kKT * kUnit),
                                     sdesc(sx + kk * kUnit, kUnit, kKT * kUnit), idesc, h > 0 || kk > 0 ? 1u : 0u);
                        mma_commit(empty(slot));
                    }
                    if (!ok) break;
                    mma_commit(tfull(buf));
                }
            }
            // every MMA issued has completed before tensor memory is released
            mma_commit(drain);
            const unsigned long long t0 = globaltimer();
            while (!mbar_try(drain, 0u))
                if (globaltimer() - t0 > kWaitNs) {
                    atomicCAS(p.err, 0, 6);
                    break;
                }
        }
    } else {
        // ---- epilogue: four warps for each 8 atoms j.  Thread row m = 8 ii + 4 h + r of an accumulator
        // (h: hi, lo).  The partial accumulators of a tile are added here in float32 (rounded to
        // nearest), then the {hi, lo} cross terms are combined and the blocks of C written.  The hi and
        // the lo columns of a row c change places from one accumulator to the next, so that each of
        // their two sums takes half of the large terms: rounding then loses 0.7 of what it takes
        // from one sum of all of them.
        const int quad = warp & 3, part = (warp - kEpiWarp) >> 2;
        const int m = 32 * quad + lane;
        const int ii = m >> 3, h = (m >> 2) & 1, r = m & 3;
        const uint32_t tlane = tmem + ((uint32_t)(32 * quad) << 16) + 64u * part;
        int it = 0;
        bool ok = true;
        int t_n = q0 < q1 ? __ldg(p.order + q0) : 0, nk_n = q0 < q1 ? __ldg(p.tile_nk + t_n) : 0;
        float zero = 0.f;
        const float least = FL == 1 ? least_sum(p.range, p.log_terms, &zero) : 0.f;
        for (int q = q0; q < q1 && ok; ++q) {
            const int t = t_n, ngr = nk_n / (FL * kKT / NB);
            if (q + 1 < q1) {
                t_n = __ldg(p.order + q + 1);
                nk_n = __ldg(p.tile_nk + t_n);
            }
            float acc[64];
#pragma unroll
            for (int e = 0; e < 64; ++e) acc[e] = 0.f;
            for (int gr = 0; gr < ngr; ++gr, ++it) {
                const int buf = it % kBufs;
                ok = mbar_wait(tfull(buf), (uint32_t)(it / kBufs) & 1u, abort_flag, p.err, 4, p.wait_ns);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                const uint32_t at = tlane + (uint32_t)(buf * kBufCols) + 4u * (gr & 1);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    uint32_t v[4], w[4];
                    tmem_ld4(at + 8u * u, v);
                    tmem_ld4((at ^ 4u) + 8u * u, w);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        acc[8 * u + e] += __uint_as_float(v[e]);
                        acc[8 * u + 4 + e] += __uint_as_float(w[e]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty(buf));
            }
            if (!ok) break;
            // columns 8 jj + 4 h' + c: hi (h' = 0) or lo (h' = 1) rows c of X_jk; rows hi and lo of the
            // same (i, r) are lanes l and l + 4: lane h = 0 finishes the first four atoms j, lane
            // h = 1 the others
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float w[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float lo = acc[8 * u + c] + acc[8 * u + 4 + c], up = acc[32 + 8 * u + c] + acc[36 + 8 * u + c];
                    // hi rows first, whichever lane adds
                    const float mine = h ? up : lo, other = __shfl_xor_sync(0xffffffffu, h ? lo : up, 4);
                    w[c] = h ? other + mine : mine + other;
                }
                const int jj = 8 * part + 4 * h + u;
                // (a block that no stored pair of blocks adds to is -2 - cp)
                const int at_c = p.cpos[(int64_t)(kGI * kJ / (NB * NB)) * t + (kJ / NB) * (ii / NB) + jj / NB];
                const int cp = at_c < -1 ? -2 - at_c : at_c;
                const int b = NB == 1 ? 4 : p.b;
                const int row = 4 * (ii % NB) + r, col = 4 * (jj % NB);
                if constexpr (FL == 1) {
                    // sums that are no numbers (a zero for an absent block may have met an infinity)
                    // or too small: FMA takes the unit
                    bool odd = false;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (NB == 1 || (row < b && col + c < b)) {
                            const float v = fabsf(w[c]);
                            odd = odd || !((v >= least || v <= zero) && v <= 3.402823466e38f);
                        }
                    const unsigned rows = __ballot_sync(0xffffffffu, odd) >> (lane & 28) & 15u;
                    if (rows != 0 && at_c >= 0) {
                        if (r == 0)
                            p.list[atomicAdd(p.count, 1)] = make_int2(((p.tile_i0[t] + ii / NB) * NB + ii % NB) * NB + jj % NB, cp);
                        continue;
                    }
                }
                if (cp < 0) continue;
                if (NB > 1 && row >= b) continue;
                if (at_c < -1) w[0] = w[1] = w[2] = w[3] = 0.f;  // also where zeros met an infinity
                float *dst = p.C + (int64_t)(b * b) * cp + row * b + col;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    if (NB > 1 && col + c >= b) continue;
                    w[c] *= p.alpha;
                    if (p.beta != 0.f) w[c] = fmaf(p.beta, dst[c], w[c]);
                    if (NB > 1 || !p.c_vec) dst[c] = w[c];
                }
                if (NB == 1 && p.c_vec) *reinterpret_cast<float4 *>(dst) = make_float4(w[0], w[1], w[2], w[3]);
                if (p.c_tm) {
                    // symmetric result: column r of the mirrored block C_ji is row r of C_ij
                    const int64_t qc = p.c_tm[cp];
                    if (qc != cp) {
                        float *mr = p.C + (int64_t)(b * b) * qc + col * b + row;
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (NB == 1 || col + c < b) mr[c * b] = w[c];
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

constexpr size_t kSmemBytes = (size_t)kStages * kStageBytes + kRingBytes + 256;

}  // namespace

TcTile tc_tile(int kind, int nb) {
    if (kind == 0) return TcTile{0, nb, kG / nb, kJT / nb, kKS / nb, kRecK / nb};
    return TcTile{1, nb, kGI / nb, kJ / nb, kKS / nb, kKT / nb};
}

int tc_plan_get(lsq_geom g, int ra, int rb, int rc, int upper, const TcTile &tile, TcPlan **out, cudaStream_t s,
                const TcRule *rule) {
    std::lock_guard<std::recursive_mutex> hold(g->mx);
    auto key = tc_plan_key(ra, rb, rc, upper, tile.kind, tile.nb);
    const int G = tile.G, JT = tile.JT, KS = tile.KS, rec = (G + JT) * tile.RK;
    auto f = g->tcplans.find(key);
    if (f != g->tcplans.end()) {
        *out = &f->second;
        return LSQ_OK;
    }
    const Pattern &PA = g->pats[ra], &PX = g->pats[rb], &PC = g->pats[rc];
    const int n = g->n;
    if (PA.max_row >= 65535 || PX.max_row >= 65535 || PC.max_row >= 65535)
        return set_error(LSQ_ERR_UNSUPPORTED, "row too long for a tensor-core plan");
    if (PC.nnzb >= ((int64_t)1 << 31) || PA.nnzb >= ((int64_t)1 << 31) || PX.nnzb >= ((int64_t)1 << 31))
        return set_error(LSQ_ERR_UNSUPPORTED, "matrix too large for a tensor-core plan (2^31 blocks)");
    const int W = (n + 31) / 32;
    const size_t smem_tiles = (size_t)3 * W * sizeof(uint32_t);
    const size_t smem_fill = (size_t)2 * W * sizeof(uint32_t) + (size_t)n * sizeof(uint16_t) + 16;
    if (std::max(smem_tiles, smem_fill) + 1024 > g->smem_optin)
        return set_error(LSQ_ERR_UNSUPPORTED, "too many atoms for the tensor-core plan builder");
    TcPlan p;
    p.upper = upper;
    p.ngroups = (n + G - 1) / G;
    *out = nullptr;
    LSQ_TRY(plan_count_triples(g, ra, rb, rc, upper, &p.triples, s));
    if (rule && !rule->can((double)p.triples)) return LSQ_OK;
    const int ng = p.ngroups;
    TcBuild a{};
    a.n = n;
    a.ngroups = ng;
    a.upper = upper;
    a.tile = tile;
    a.a_ptr = PA.row_ptr.p;
    a.a_col = PA.col.p;
    a.x_ptr = PX.row_ptr.p;
    a.x_col = PX.col.p;
    a.c_ptr = PC.row_ptr.p;
    a.c_col = PC.col.p;
    const int grid = std::max(1, std::min(ng, g->num_sms * 2));
    // pass 1: tiles per group
    std::vector<int32_t> nt(std::max(ng, 1), 0), toff(ng + 1, 0);
    if (ng > 0) {
        DevBuf<int32_t> nt_d;
        LSQ_TRY(nt_d.alloc(ng));
        LSQ_CUDA_TRY(cudaFuncSetAttribute(k_tc_groups, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)(W * sizeof(uint32_t))));
        note_launch();
        k_tc_groups<<<grid, 512, W * sizeof(uint32_t), s>>>(a, nt_d.p);
        LSQ_CHECK_LAUNCH();
        LSQ_CUDA_TRY(cudaMemcpyAsync(nt.data(), nt_d.p, sizeof(int32_t) * ng, cudaMemcpyDeviceToHost, s));
        LSQ_CUDA_TRY(cudaStreamSynchronize(s));
    }
    for (int q = 0; q < ng; ++q) toff[q + 1] = toff[q] + nt[q];
    p.ntiles = toff[ng];
    const int T = std::max(p.ntiles, 1);
    DevBuf<int32_t> toff_d;
    LSQ_TRY(toff_d.alloc(ng + 1));
    LSQ_TRY(p.tile_j.alloc((size_t)JT * T));
    LSQ_TRY(p.tile_i0.alloc(T));
    LSQ_TRY(p.tile_nk.alloc(T));
    LSQ_TRY(p.tile_posoff.alloc(T));
    LSQ_TRY(p.cpos.alloc((size_t)G * JT * T));
    std::vector<int32_t> tnk(T, 0);
    std::vector<int64_t> tpo(T, 0), tko(T, 0);
    int64_t total = 0, klen = 0;
    p.grid = std::max(1, std::min(p.ntiles, g->num_sms));
    std::vector<int32_t> cst(p.grid, 0), order(T, 0), first(p.grid + 1, 0);
    std::vector<int64_t> rec0(p.grid, 0);
    if (p.ntiles > 0) {
        LSQ_CUDA_TRY(cudaMemcpyAsync(toff_d.p, toff.data(), sizeof(int32_t) * (ng + 1), cudaMemcpyHostToDevice, s));
        a.g_toff = toff_d.p;
        a.tile_j = p.tile_j.p;
        a.tile_nk = p.tile_nk.p;
        // pass 2: atoms j of the tiles, k-list lengths
        LSQ_CUDA_TRY(cudaFuncSetAttribute(k_tc_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_tiles));
        note_launch();
        k_tc_tiles<<<grid, 512, smem_tiles, s>>>(a);
        LSQ_CHECK_LAUNCH();
        LSQ_CUDA_TRY(cudaMemcpyAsync(tnk.data(), p.tile_nk.p, sizeof(int32_t) * p.ntiles, cudaMemcpyDeviceToHost, s));
        LSQ_CUDA_TRY(cudaStreamSynchronize(s));
        // tiles in order, each to the CTA with the least work so far: neighbouring tiles, which share
        // rows, run at about the same time, and the loads differ by no more than a tile.  A CTA's
        // stage records follow one another in its stream.
        std::vector<std::vector<int32_t>> mine(p.grid);
        std::priority_queue<std::pair<int64_t, int>, std::vector<std::pair<int64_t, int>>, std::greater<>> load;
        for (int c = 0; c < p.grid; ++c) load.emplace(0, c);
        for (int t = 0; t < p.ntiles; ++t) {
            auto [w, c] = load.top();
            load.pop();
            mine[c].push_back(t);
            load.emplace(w + tnk[t] / KS + 2, c);  // the last lines of a tile cost about two groups
        }
        int q = 0;
        for (int c = 0; c < p.grid; ++c) {
            first[c] = q;
            rec0[c] = total;
            for (int t : mine[c]) {
                order[q++] = t;
                tpo[t] = total;
                total += (int64_t)rec * (tnk[t] / tile.RK);
                cst[c] += tnk[t] / KS;
            }
        }
        first[p.grid] = q;
        for (int t = 0; t < p.ntiles; ++t) {
            tko[t] = klen;
            klen += tnk[t];
            p.units += (int64_t)(G + JT) * tnk[t];
            p.max_nk = std::max(p.max_nk, tnk[t]);
            p.dense_triples += (int64_t)G * JT * tnk[t];
        }
    }
    if (rule && !rule->pays(p)) return LSQ_OK;
    LSQ_TRY(p.pos.alloc(std::max<int64_t>(total, 16)));
    LSQ_TRY(p.cta_stages.alloc(p.grid));
    LSQ_TRY(p.order.alloc(T));
    LSQ_TRY(p.cta_first.alloc(p.grid + 1));
    LSQ_TRY(p.cta_rec.alloc(p.grid));
    LSQ_CUDA_TRY(cudaMemcpyAsync(p.order.p, order.data(), sizeof(int32_t) * T, cudaMemcpyHostToDevice, s));
    LSQ_CUDA_TRY(cudaMemcpyAsync(p.cta_first.p, first.data(), sizeof(int32_t) * (p.grid + 1), cudaMemcpyHostToDevice, s));
    LSQ_CUDA_TRY(cudaMemcpyAsync(p.cta_rec.p, rec0.data(), sizeof(int64_t) * p.grid, cudaMemcpyHostToDevice, s));
    LSQ_CUDA_TRY(cudaMemcpyAsync(p.cta_stages.p, cst.data(), sizeof(int32_t) * p.grid, cudaMemcpyHostToDevice, s));
    std::vector<int32_t> ti0(T, 0);
    for (int q = 0; q < ng; ++q)
        for (int t = toff[q]; t < toff[q + 1]; ++t) ti0[t] = G * q;
    LSQ_CUDA_TRY(cudaMemcpyAsync(p.tile_i0.p, ti0.data(), sizeof(int32_t) * T, cudaMemcpyHostToDevice, s));
    if (p.ntiles > 0) {
        DevBuf<int32_t> klist;
        DevBuf<int64_t> tko_d;
        LSQ_TRY(klist.alloc(std::max<int64_t>(klen, 1)));
        LSQ_TRY(tko_d.alloc(p.ntiles));
        LSQ_CUDA_TRY(cudaMemcpyAsync(p.tile_posoff.p, tpo.data(), sizeof(int64_t) * p.ntiles, cudaMemcpyHostToDevice, s));
        LSQ_CUDA_TRY(cudaMemcpyAsync(tko_d.p, tko.data(), sizeof(int64_t) * p.ntiles, cudaMemcpyHostToDevice, s));
        a.tile_posoff = p.tile_posoff.p;
        a.tile_koff = tko_d.p;
        a.klist = klist.p;
        a.pos = p.pos.p;
        a.cpos = p.cpos.p;
        // pass 3: k-lists, block offsets, positions in C
        LSQ_CUDA_TRY(cudaFuncSetAttribute(k_tc_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_fill));
        note_launch();
        k_tc_fill<<<grid, 512, smem_fill, s>>>(a);
        LSQ_CHECK_LAUNCH();
        static_assert(kG + kJT <= kMaxRows && kG * kJT <= kMaxPairs && kMaxPairs % 256 == 0, "tiles of k_tc_empty");
        note_launch();
        k_tc_empty<<<std::min(p.ntiles, g->num_sms * 8), 256, 0, s>>>(a, p.ntiles);
        LSQ_CHECK_LAUNCH();
        // blocks the launches copy (the other slots are zeros stored in shared memory)
        DevBuf<unsigned long long> cnt;
        LSQ_TRY(cnt.alloc(1));
        LSQ_CUDA_TRY(cudaMemsetAsync(cnt.p, 0, sizeof(unsigned long long), s));
        note_launch();
        k_count_present<<<std::max(1, std::min<int>((int)((total + 255) / 256), g->num_sms * 8)), 256, 0, s>>>(
            total, p.pos.p, cnt.p);
        LSQ_CHECK_LAUNCH();
        unsigned long long h = 0;
        LSQ_CUDA_TRY(cudaMemcpyAsync(&h, cnt.p, sizeof(h), cudaMemcpyDeviceToHost, s));
        LSQ_CUDA_TRY(cudaStreamSynchronize(s));  // the scratch lists are freed on return
        p.present = (int64_t)h;
    }
    if (std::getenv("LSQ_TC_LOG")) {
        const int smax = p.grid > 0 ? *std::max_element(cst.begin(), cst.end()) : 0;
        std::fprintf(stderr,
                     "lsq tc plan: ranges (%g, %g, %g) tri %d: %d tiles, %lld blocks gathered, %lld dense / %lld "
                     "triples (%.3f), %d CTAs, max %d stages per CTA, records %.1f MB\n",
                     PA.R, PX.R, PC.R, upper, p.ntiles, (long long)p.units, (long long)p.dense_triples,
                     (long long)p.triples, p.dense_triples ? (double)p.triples / p.dense_triples : 0.0, p.grid, smax,
                     4.0 * total / 1e6);
    }
    *out = &g->tcplans.emplace(key, std::move(p)).first->second;
    return LSQ_OK;
}

namespace {

// mode: 0 X, 1 X^T, 2 X + X^T (see k_split_tf32).
int split_operand(lsq_geom g, int b, int nb, int r, int mode, const float *X, char *buf, unsigned *range, uint8_t *any,
                  cudaStream_t s) {
    const int64_t nnzb = g->pats[r].nnzb, units = nnzb * nb * nb;
    if (nnzb == 0) return LSQ_OK;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((units * 4 + 255) / 256, (int64_t)g->num_sms * (range ? 8 : 32)));
    const bool vec = reinterpret_cast<uintptr_t>(X) % 16 == 0;
    auto go = [&](auto kern) {
        kern<<<blocks, 256, 0, s>>>(nnzb, b, g->pats[r].tmap.p, X, vec, reinterpret_cast<float4 *>(buf), range, any);
    };
    note_launch();
    if (nb == 1) go(mode == 1 ? k_split_tf32<1, 1> : (mode == 2 ? k_split_tf32<2, 1> : k_split_tf32<0, 1>));
    else go(mode == 1 ? k_split_tf32<1, 4> : (mode == 2 ? k_split_tf32<2, 4> : k_split_tf32<0, 4>));
    LSQ_CHECK_LAUNCH();
    return LSQ_OK;
}

}  // namespace

thread_local bool g_fma_products = false;
thread_local SplitStore *g_split_store = nullptr;

SplitLock::SplitLock(lsq_geom g, cudaStream_t s) : g_(g), s_(s), lock_(g->mx, std::defer_lock) {
    auto check = [&](cudaError_t e) {
        if (e != cudaSuccess && rc_ == LSQ_OK)
            rc_ = set_error(LSQ_ERR_CUDA, std::string("ordering the split buffers: ") + cudaGetErrorString(e));
    };
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    check(cudaStreamIsCapturing(s, &st));
    capturing_ = st != cudaStreamCaptureStatusNone;
    store_ = capturing_ ? g_split_store : &g->split;
    if (capturing_ || rc_ != LSQ_OK) return;
    lock_.lock();
    unsigned long long id = 0;
    check(cudaStreamGetId(s, &id));
    if (!g->split_ev) check(cudaEventCreateWithFlags(&g->split_ev, cudaEventDisableTiming));
    if (rc_ != LSQ_OK) return;
    if (g->split_used && g->split_stream != id) check(cudaStreamWaitEvent(s, g->split_ev, 0));
    g->split_stream = id;
}

SplitLock::~SplitLock() {
    if (graph_mem_) cudaFreeAsync(graph_mem_, s_);  // a product that failed half-way
}

int SplitLock::buffers(const SplitSizes &need, SplitBuffers *out) {
    auto has = [](const auto &buf, size_t bytes) { return buf.n * sizeof(*buf.p) >= bytes; };
    if (capturing_ && store_ &&
        !(has(store_->a, need.a) && has(store_->x, need.x) && has(store_->ai, need.ai) && has(store_->xi, need.xi) &&
          has(store_->list, need.list)))
        store_ = nullptr;
    if (store_) {
        auto grow = [&](auto &buf, size_t bytes) { return has(buf, bytes) ? LSQ_OK : buf.alloc(bytes / sizeof(*buf.p)); };
        if (!has(store_->a, need.a)) store_->a_src = nullptr;
        LSQ_TRY(grow(store_->a, need.a));
        LSQ_TRY(grow(store_->x, need.x));
        LSQ_TRY(grow(store_->ai, need.ai));
        LSQ_TRY(grow(store_->xi, need.xi));
        LSQ_TRY(grow(store_->list, need.list));
        out->a = store_->a.p;
        out->x = store_->x.p;
        out->ai = store_->ai.p;
        out->xi = store_->xi.p;
        out->list = store_->list.p;
        return LSQ_OK;
    }
    const size_t size[5] = {need.a, need.x, need.ai, need.xi, need.list};
    size_t total = 0;
    for (size_t n : size) total += (n + 255) / 256 * 256;
    const cudaError_t e = cudaMallocAsync(&graph_mem_, total, s_);
    if (e != cudaSuccess) {
        graph_mem_ = nullptr;
        return set_error(LSQ_ERR_OOM, std::string("memory of a captured product: ") + cudaGetErrorString(e));
    }
    char *p[5], *q = static_cast<char *>(graph_mem_);
    for (int k = 0; k < 5; q += (size[k] + 255) / 256 * 256, ++k) p[k] = q;
    out->a = p[0];
    out->x = p[1];
    out->ai = reinterpret_cast<int *>(p[2]);
    out->xi = reinterpret_cast<int *>(p[3]);
    out->list = reinterpret_cast<int *>(p[4]);
    return LSQ_OK;
}

int SplitLock::release() {
    if (capturing_) {
        void *m = graph_mem_;
        graph_mem_ = nullptr;
        if (m) LSQ_CUDA_TRY(cudaFreeAsync(m, s_));
        return LSQ_OK;
    }
    LSQ_CUDA_TRY(cudaEventRecord(g_->split_ev, s_));
    g_->split_used = true;
    return LSQ_OK;
}

int dev_err_ptr(lsq_geom g, int **out) {
    std::lock_guard<std::recursive_mutex> hold(g->mx);
    LSQ_TRY(pinned_words(g));
    *out = reinterpret_cast<int *>(g->red.host + kPinned);
    return LSQ_OK;
}

int pinned_words(lsq_geom g) {
    std::lock_guard<std::recursive_mutex> hold(g->mx);
    if (g->red.host) return LSQ_OK;
    double *p = nullptr;
    LSQ_CUDA_TRY(cudaMallocHost(&p, sizeof(double) * (kPinned + 1)));
    p[kPinned] = 0.0;
    g->red.host = p;
    return LSQ_OK;
}

int waits_ok(lsq_geom g) {
    std::lock_guard<std::recursive_mutex> hold(g->mx);
    if (!g->red.host) return LSQ_OK;
    volatile int *word = reinterpret_cast<int *>(g->red.host + kPinned);
    const int h = *word;
    if (h == 0) return LSQ_OK;
    *word = 0;
    static const char *where[] = {"", "copy issue (stage free)", "MMA issue (stage full)", "MMA issue (accumulator free)",
                                  "epilogue (accumulator full)", "copies in flight at exit", "MMAs in flight at exit"};
    return set_error(LSQ_ERR_TIMEOUT, std::string("a bounded wait of the tensor-core product expired: ") +
                                          (h > 0 && h < 7 ? where[h] : "unknown"));
}

int split_choice(lsq_geom g, int b, int ra, int rb, int rc, int upper, bool *use, cudaStream_t s) {
    *use = false;
    const int nb = slice_units(b);
    if (nb == 0 || g_fma_products || g_group_rec || g->n == 0 || std::getenv("LSQ_PLAN_VARIANT")) return LSQ_OK;
    // LSQ_F32_SPLIT fixes the choice (0 FMA, 1 split TF32), for tests
    const char *fixed = std::getenv("LSQ_F32_SPLIT");
    if (fixed && std::atoi(fixed) == 0) return LSQ_OK;
    const int64_t blocks = g->pats[ra].nnzb + g->pats[rb].nnzb;
    if ((size_t)kUnit * nb * nb * (size_t)blocks > g->mem_total / 8) return LSQ_OK;  // see sliced_choice
    // The FMA schedules take 10 to 13 ps a triple of 4 x 4 blocks (13 TFLOP/s for larger ones), this
    // kernel 1.2 ps a dense triple of units, 0.04 ns a block split and 9 us more for its launches.
    // Measured, FMA against split: 989 atoms, triples 76 M of 273 M dense, 781 and 401 us; 42 of 210 M,
    // 393 and 291 us; 9.7 of 162 M, 161 and 230 us; 512 atoms, 9.8 of 85 M, 121 and 129 us; 64 atoms,
    // 0.26 of 0.26 M, 17 and 25 us; 493 atoms of 13 x 13 blocks, 22 M triples, 7138 and 4040 us.  Error
    // where it takes over (216 to 4096 atoms, 26 to 929 triples a block): the 2-norm 1.2 to 3.8 times
    // smaller than FMA's, the largest of an element relative to its sum of |a| |b| 1.4 to 6 times
    // (2.7e-7 against 7.3e-7 for SL.Q^T of 4096 atoms).  Lists of less than 16 triples a block stay
    // with FMA: their sums are too short for its rounding to exceed the split's.
    const double fma_ps = nb == 1 ? 10.5 : 2.0 * b * b * b / 13.0, tc_ps = 1.2 * nb * nb * nb;
    const double split_ps = 40.0 * blocks * nb * nb + 9e6;
    const double c_blocks = (upper ? 0.5 : 1.0) * (double)g->pats[rc].nnzb;
    TcRule rule;
    // (a product has at least as many dense triples as stored ones)
    rule.can = [=](double n) { return n * (fma_ps - tc_ps) > split_ps && n >= 16 * c_blocks; };
    rule.pays = [=](const TcPlan &p) {
        return p.triples >= 16 * c_blocks && p.triples * fma_ps > p.dense_triples * tc_ps + split_ps;
    };
    return tensor_choice(g, ra, rb, rc, upper, tc_tile(1, nb), fixed != nullptr, rule, nullptr, use, s);
}

int tensor_choice(lsq_geom g, int ra, int rb, int rc, int upper, const TcTile &tile, bool fixed, const TcRule &rule,
                  TcPlan **plan, bool *use, cudaStream_t s) {
    *use = false;
    std::lock_guard<std::recursive_mutex> hold(g->mx);
    const auto key = tc_plan_key(ra, rb, rc, upper, tile.kind, tile.nb);
    const Pattern &PA = g->pats[ra], &PX = g->pats[rb], &PC = g->pats[rc];
    if (!fixed) {
        const auto known = g->tc_use.find(key);
        if (known != g->tc_use.end() && !known->second) return LSQ_OK;
        // the longest lists there can be settle it for small systems, without a plan
        if (known == g->tc_use.end() &&
            !rule.can((upper ? 0.5 : 1.0) * (double)PC.nnzb * std::min(PA.max_row, PX.max_row) + g->n)) {
            g->tc_use[key] = false;
            return LSQ_OK;
        }
    }
    TcPlan *p = nullptr;
    const int rc2 = tc_plan_get(g, ra, rb, rc, upper, tile, &p, s, fixed ? nullptr : &rule);
    if (rc2 == LSQ_ERR_OOM || rc2 == LSQ_ERR_UNSUPPORTED) {
        (void)cudaGetLastError();
        clear_error();
        p = nullptr;
    } else {
        LSQ_TRY(rc2);
    }
    *use = p && p->ntiles > 0 && (fixed || rule.pays(*p));
    if (!fixed) g->tc_use[key] = *use;
    if (plan) *plan = p;
    return LSQ_OK;
}

int tc_block_matmul(lsq_geom g, int ra, int ta, const float *A, int rb, int tb, const float *B, int rc, float *C,
                    double alpha, double beta, int upper, bool mirror, int64_t *triples, cudaStream_t s,
                    bool b_sym, bool reuse_a, int b, bool f32, bool *done) {
    LSQ_TRY(ensure_tmap(g, ra, s));
    LSQ_TRY(ensure_tmap(g, rb, s));
    const int nb = slice_units(b);
    if (done) *done = true;
    if (nb == 0 || (!f32 && nb != 1)) return set_error(LSQ_ERR_INVALID_ARG, "internal: block size of a tensor-core product");
    TcPlan *p = nullptr;
    LSQ_TRY(tc_plan_get(g, ra, rb, rc, upper, tc_tile(1, nb), &p, s));
    if (triples) *triples = p->triples;
    if (g->n == 0 || g->pats[rc].nnzb == 0 || p->ntiles == 0) return LSQ_OK;
    if (!p->pos.p || !p->cpos.p || !p->tile_nk.p || !p->cta_rec.p || !p->order.p || !p->cta_stages.p)
        return set_error(LSQ_ERR_CUDA, "tensor-core plan without its records");
    if (upper == 1 && mirror) LSQ_TRY(ensure_tmap(g, rc, s));
    SplitLock lock(g, s);
    LSQ_TRY(lock.status());
    SplitSizes need;
    need.a = (size_t)kUnit * nb * nb * (size_t)std::max<int64_t>(g->pats[ra].nnzb, 1);
    need.x = (size_t)kUnit * nb * nb * (size_t)std::max<int64_t>(g->pats[rb].nnzb, 1);
    // (float32: the number of listed units, the words of k_split_tf32, four an operand, the units)
    constexpr int kHead = 12;
    auto unit_bytes = [&](int r) { return f32 ? ((size_t)nb * nb * (size_t)g->pats[r].nnzb + 3) / 4 * 4 : 0; };
    need.ai = unit_bytes(ra);
    need.xi = unit_bytes(rb);
    need.list = f32 ? sizeof(int) * (kHead + 2 * (size_t)nb * nb * (size_t)g->pats[rc].nnzb) : 0;
    SplitBuffers sb;
    const int got = lock.buffers(need, &sb);
    if (done) *done = got == LSQ_OK;
    if (done && got == LSQ_ERR_OOM) {
        (void)cudaGetLastError();
        clear_error();
        return LSQ_OK;
    }
    LSQ_TRY(got);
    unsigned *range = f32 ? reinterpret_cast<unsigned *>(sb.list) + 4 : nullptr;
    if (f32) LSQ_CUDA_TRY(cudaMemsetAsync(sb.list, 0, kHead * sizeof(int), s));
    uint8_t *a_any = f32 ? reinterpret_cast<uint8_t *>(sb.ai) : nullptr, *x_any = f32 ? reinterpret_cast<uint8_t *>(sb.xi) : nullptr;
    // op(A) and X = op(B)^T (B's rows when trans_b, else B read through its transpose map; B +
    // B^T when b_sym) in split form, in buffers held by g.  The split of A is kept when the
    // caller says A is unchanged since the previous split of the same array (a float32 product needs
    // the range of its values too, so it splits A again).
    SplitStore *st = lock.store();
    const bool keep = !f32 && reuse_a && st && st->holds(A, ra, ta != 0, false);
    const int bmode = b_sym ? 2 : (tb == 0 ? 1 : 0);
    if (!keep) {
        if (st) st->a_src = nullptr;
        LSQ_TRY(split_operand(g, b, nb, ra, ta != 0 ? 1 : 0, A, sb.a, range, a_any, s));
        if (st) st->set(A, ra, ta != 0, false);
    }
    LSQ_TRY(split_operand(g, b, nb, rb, bmode, B, sb.x, range ? range + 4 : nullptr, x_any, s));
    int *err = nullptr;
    LSQ_TRY(dev_err_ptr(g, &err));
    TcArgs a;
    a.b = b;
    a.c_vec = reinterpret_cast<uintptr_t>(C) % 16 == 0;
    a.order = p->order.p;
    a.cta_first = p->cta_first.p;
    a.tile_nk = p->tile_nk.p;
    a.cpos = p->cpos.p;
    a.cta_rec = p->cta_rec.p;
    a.cta_stages = p->cta_stages.p;
    a.pos = p->pos.p;
    a.As = sb.a;
    a.Xs = sb.x;
    a.C = C;
    a.c_tm = upper == 1 && mirror ? g->pats[rc].tmap.p : nullptr;
    a.alpha = (float)alpha;
    a.beta = (float)beta;
    a.range = range;
    a.count = sb.list;
    a.list = reinterpret_cast<int2 *>(sb.list + kHead);
    a.tile_i0 = p->tile_i0.p;
    a.log_terms = 2;
    while ((1 << a.log_terms) < 4 * nb * p->max_nk) ++a.log_terms;
    a.err = err;
    // LSQ_TC_WAIT_NS lowers the bound of the pipeline waits (0: any wait that does not succeed at
    // once expires), so that a test can check the timeout path and its status; default 1 s
    a.wait_ns = kWaitNs;
    if (const char *w = std::getenv("LSQ_TC_WAIT_NS")) a.wait_ns = std::strtoull(w, nullptr, 10);
    const auto product = !f32 ? k_tc_product<1, 2> : (nb == 1 ? k_tc_product<1, 1> : k_tc_product<4, 1>);
    LSQ_CUDA_TRY(cudaFuncSetAttribute(product, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes));
    note_launch();
    product<<<p->grid, kThreads, kSmemBytes, s>>>(a);
    LSQ_CHECK_LAUNCH();
    // (a symmetric result's lower blocks are written by the kernel itself, see c_tm)
    if (f32)
        LSQ_TRY(launch_listed(g, b, nb, ra, ta, A, rb, bmode, B, rc, C, alpha, beta, a.c_tm, a.count, a.list, s,
                              {a_any, x_any, nullptr, nullptr, range + 2, range + 6}));
    return lock.release();
}

}  // namespace lsq

using namespace lsq;

extern "C" int lsq_product_plan_info(lsq_geom g, int range_a, int range_b, int range_c, int triangle,
                                     int64_t *info_host) {
    clear_error();
    LSQ_TRY(geom_check(g, range_a));
    LSQ_TRY(geom_check(g, range_b));
    LSQ_TRY(geom_check(g, range_c));
    if (!info_host) return set_error(LSQ_ERR_INVALID_ARG, "info_host is null");
    if (triangle < 0 || triangle > 3) return set_error(LSQ_ERR_INVALID_ARG, "triangle must be 0..3");
    const int upper = triangle == 3 ? 2 : (triangle >= 1 ? 1 : 0);
    std::lock_guard<std::recursive_mutex> hold(g->mx);
    const auto key = std::make_tuple(range_a, range_b, range_c + 1000 * upper);
    auto f = g->tcplans.find(tc_plan_key(range_a, range_b, range_c, upper, 1, 1));
    if (f == g->tcplans.end()) f = g->tcplans.find(tc_plan_key(range_a, range_b, range_c, upper, 0, 1));
    auto ch = g->tc_choice.find(key);
    if (f == g->tcplans.end() && ch == g->tc_choice.end())
        return set_error(LSQ_ERR_INVALID_ARG, "no tensor-core plan or choice for these ranges yet");
    for (int k = 0; k < 6; ++k) info_host[k] = -1;
    if (f != g->tcplans.end()) {
        const TcPlan &p = f->second;
        info_host[0] = p.triples;
        info_host[1] = p.dense_triples;
        info_host[2] = p.units;
        info_host[3] = p.ntiles;
        info_host[5] = p.present;
    }
    info_host[4] = ch == g->tc_choice.end() ? -1 : ch->second;
    return LSQ_OK;
}

extern "C" int lsq_device_status(lsq_geom g, void *stream) {
    clear_error();
    if (!g) return set_error(LSQ_ERR_INVALID_ARG, "null geometry");
    if (!g->red.host) return LSQ_OK;  // no product with bounded waits has run
    LSQ_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    return waits_ok(g);
}

// Float64 truncated block products on the tensor cores, from exact integer slices (4 x 4 blocks, and
// blocks of 9 to 16 as 4 x 4 units of them).
//
// Sec. 2.3.2 of the paper: C_ij = sum_k A_ik B_kj over the stored blocks (i, j) of C.  The FP64
// pipe of this GPU (1.25 TFLOP/s measured) bounds the FMA kernels of such a product, while its
// 16-bit tensor cores are 1500 times faster.  So the operands are cut into slices whose products
// the tensor cores form without rounding (the error-free splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59, 2012):
//
//  * Slices.  A scalar row (atom, orbital) of op(A) and of X = op(B)^T gets a power-of-two scale
//    2^e above its largest entry; v 2^-e is held to 90 bits as ten balanced digits in base 512,
//    v = 2^e sum_d q_d 512^(9-d) 2^-89, -256 <= q_d <= 256.  Each digit is exact in bf16, and the
//    product of two is an integer of at most 2^16.
//  * Orders.  A product of digits a and b has weight 512^-(a+b).  Those of one order a + b are
//    summed by the tensor cores in float32: a tile's 16 atoms k give at most 256 products to any
//    accumulator of orders 0 to 7, so those sums are integers of at most 2^24, and exact.  (Orders
//    8 and 9 get up to 320.  A sum of theirs beyond 2^24, for which nearly all digits have to be at
//    their bound, loses its last bit, no more than what is left out.)  Orders 0 to 9 are kept in
//    full and five of the nine products of order 10; what is left out of a sum of n products is
//    2^-91 sqrt(n) of a row's largest entry times a column's.
//  * Sums.  The accumulators of 16 atoms k are added to 64-bit integers, orders 0-3 in units of
//    order 3, 4-7 in units of order 7, 8 and 9 in units of order 9.  16 atoms k add at most
//    2^49 + 2^41 to the first and 3 2^49 + 2^42 to the second, so all stay below 2^62 over kMaxGroups
//    of them.  They are put together in 128 bits: the only rounding of a result is the last one, to
//    float64.
//
// The error of a sum is thus relative to the row's and the column's largest entries, and on decaying
// matrices many sums lie far below these.  A sum 2^-33 or so below them (see kLeastBits), in a row or
// column with entries small enough for all its terms to be as small, could be off by more than its
// FP64 sum.  The block it belongs to is not written: it is listed and summed by k_listed in
// FP64, as is every block of a row that holds an infinity or NaN.  So every element is as accurate as
// its FP64 sum.  (Eight digits would take two thirds of the time, but would have to leave 87 % of the
// blocks of LSL at 1728 atoms to FP64; ten leave some 5 % there and 1 % in most products.)
//
// The kernel is the gathered-panel tcgen05 kernel of tc.cu (same plan, same roles) on 320-byte
// units.  A unit of block (i, k) holds, for each pair t of digits (2t, 2t + 1) and each column kk
// of the block, 16 bytes: the four rows of digit 2t, the four rows of digit 2t + 1.  That is one
// K-row of an MN-major core matrix (8 M x 8 K), two atoms k fill it, and the two digits and four
// rows of an atom are 8 rows (of X) or 8 columns (of A) of the accumulator.  Pair t of X times
// the pairs 0 .. 4 - t of A, side by side along N, lands in accumulator columns 64 t and up, so
// column group cp collects the pairs with t + bp = cp: two MMAs at most per t and 4 atoms k, one for
// each part of the accumulator.  Measured (LS.L of 2744 atoms, 8 digits and 10): 7.98 and 11.2 ms.
// What bounds it is the issue of the copies together with the MMAs' and the copies' traffic in shared
// memory: with the MMAs cut to a quarter it takes 9.4 ms, with every copy writing zeros 11.3.  Tried
// and slower: stages of 4 atoms k in a ring of 7 (12.8 ms), six copying warps (12.0, fewer registers
// for the sums), the 128-byte swizzle (13.2).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <string>
#include <type_traits>

#include "listed.h"
#include "lsq_internal.h"
#include "tc_ptx.h"

namespace lsq {
namespace {

constexpr int kPairs = 5;                               // pairs of digits
constexpr int kHead = 256, kTail = 64;                  // bytes of a sliced block: pairs 0-3, pair 4 (an array of each)
constexpr int kUnit = kHead + kTail;
constexpr int kKP = kRecK / 2;                          // pairs of atoms k in a stage
constexpr int kCore = 128;                              // bytes of a core matrix
constexpr int kPanelX = kPairs * kKP * kJT * kCore;     // [t][pair of k][j], 40 KB
constexpr int kPanelA = kKP * kPairs * kG * kCore;      // [pair of k][pair of digits][i], 20 KB
constexpr int kStageBytes = kPanelX + kPanelA;
constexpr int kStages = 3;
// Tensor memory, all 512 columns: an accumulator has 64 for each pair of orders.  Its upper part
// (orders 0-5) has two places, the lower part (orders 6-9), which the epilogue reads first, one.
constexpr int kUpPairs = 3;
constexpr int kUpCols = 64 * kUpPairs, kLowAt = kUpCols;
constexpr int kBufs = 2, kBufCols = 320;                // upper parts at columns 0 and 320
constexpr int kTmemCols = 512;
constexpr int kCopyWarps = 3;
constexpr int kMmaWarp = 3;
constexpr int kEpiWarp = 4;                             // warps 4-19 read the accumulator
constexpr int kEpiWarps = 16;
constexpr int kEpiI = kG / (kEpiWarps / 4);             // atoms i of one of them
constexpr int kThreads = 32 * (kEpiWarp + kEpiWarps);
constexpr int kRecRing = 16, kRecAhead = 8;             // records in shared memory
constexpr int kRingBytes = kRecRing * kRec * 4;
constexpr size_t kSmemBytes = (size_t)kStages * kStageBytes + kRingBytes + 256;

// Row information of a sliced operand, one word per scalar row: the scale exponent in the low 16
// bits (biased by 4096), kDeep if the row holds nonzero entries below 2^-kDeepBits of its scale,
// kNone if it holds no nonzero entry, kBad if it holds an infinity or a NaN.
constexpr int kExpBias = 4096;
constexpr int kDeep = 1 << 16, kBad = kBadRow, kNone = 1 << 18;
constexpr int kDeepBits = 16;
constexpr int kMaxGroups = 2048;  // groups of 16 atoms k of a tile
constexpr int kScaleBits = 106;   // full scale, the product of the two scales, in units of order 10
// Sums of n products shorter than kLeastBits + log2(n) / 2 bits are taken in FP64 where a row is deep
// (the products left out amount to 2^15.4 sqrt(n) units, 2^-54 of such a sum).
constexpr int kLeastBits = 70;

// ---- slicing ---------------------------------------------------------------------------------
struct SliceArgs {
    const int64_t *ptr;   // row pointers of the operand's pattern
    const int64_t *tm;    // its transpose map (modes 1 and 2)
    const double *X;
    uint4 *out, *tail;    // [nnzb][NB][NB][4][4] and [nnzb][NB][NB][4] 16-byte chunks
    int *info;            // [4 NB n]
    uint8_t *any;         // [nnzb][NB][NB]: 0 if the unit is all zeros
    int mode;             // 0 X, 1 X^T, 2 X + X^T
    int b;                // block size
};

// A block is NB x NB units of 4 x 4 (NB = 1: 4 x 4 blocks; NB = 4: b in 9 .. 16, zeros beyond b), unit
// (R, K) the rows 4 R .. and columns 4 K ...  Item e of block p is column 4 K + kk of the rows 4 R ..
// 4 R + 3, e = ((p NB + R) NB + K) 4 + kk; its four values:
template <int NB>
__device__ __forceinline__ void slice_load(const SliceArgs &a, int64_t p, int R, int c, double (&v)[4]) {
    if constexpr (NB == 1) {
        if (a.mode != 1) {
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = __ldg(a.X + 16 * p + 4 * r + c);
        }
        if (a.mode != 0) {
            const double2 *q = reinterpret_cast<const double2 *>(a.X + 16 * a.tm[p] + 4 * c);
            const double2 x = __ldg(q), y = __ldg(q + 1);
            const double w[4] = {x.x, x.y, y.x, y.y};
#pragma unroll
            for (int r = 0; r < 4; ++r) v[r] = a.mode == 1 ? w[r] : v[r] + w[r];
        }
    } else {
        const int b = a.b, bb = b * b;
        const double *X = a.X + (int64_t)bb * p, *Xt = a.mode ? a.X + (int64_t)bb * a.tm[p] : nullptr;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int row = 4 * R + r;
            const bool in = row < b && c < b;
            v[r] = 0.0;
            if (in && a.mode != 1) v[r] = __ldg(X + row * b + c);
            if (in && a.mode != 0) v[r] += __ldg(Xt + c * b + row);
        }
    }
}

// The digit d in [0, 511], minus 256, as the upper half of a float32 (exact in bf16).
__device__ __forceinline__ uint32_t digit_bf16(uint32_t d) {
    return __float_as_uint(__uint_as_float(0x4b000000u | d) - 8388864.0f) >> 16;
}

// One thread block per atom row (grid-stride over the rows of the first, then of the second
// operand): the largest exponent of each of the row's four scalar rows, then the digits (the
// second read of the row comes from L1 or L2).  Bound by HBM: 128 bytes read and 320 written per
// block.
template <int NB>
__global__ void __launch_bounds__(NB == 1 ? 256 : 1024) k_sl_slice(int n, SliceArgs a0, SliceArgs a1, int nops, int *__restrict__ count) {
    constexpr int kIt = 4 * NB * NB;  // items of a block; a thread's items all lie in sub-row R
    __shared__ int s_max[4 * NB], s_deep[4 * NB], s_any[4 * NB];
    const int R = NB == 1 ? 0 : (int)(threadIdx.x / (4 * NB)) % NB, c = (int)threadIdx.x % (4 * NB);
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = 0;
    for (int row = blockIdx.x; row < n * nops; row += gridDim.x) {
        const bool second = row >= n;
        const SliceArgs &a = second ? a1 : a0;
        const int i = second ? row - n : row;
        const int64_t p0 = a.ptr[i];
        const int64_t m = (a.ptr[i + 1] - p0) * kIt;
        if (threadIdx.x < 4 * NB) {
            s_max[threadIdx.x] = 0;
            s_deep[threadIdx.x] = 0;
            s_any[threadIdx.x] = 0;
        }
        __syncthreads();
        int mx[4] = {0, 0, 0, 0};
        for (int64_t e = threadIdx.x; e < m; e += blockDim.x) {
            double v[4];
            slice_load<NB>(a, p0 + e / kIt, R, c, v);
#pragma unroll
            for (int r = 0; r < 4; ++r) mx[r] = max(mx[r], (int)(((unsigned)__double2hiint(v[r]) >> 20) & 0x7ffu));
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            // (a warp spans two sub-rows R when NB = 4)
            const unsigned half = NB == 1 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);
            mx[r] = __reduce_max_sync(half, mx[r]);
            if ((threadIdx.x & (NB == 1 ? 31 : 15)) == 0) atomicMax(&s_max[4 * R + r], mx[r]);
        }
        __syncthreads();
        int deep = 0, any = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) mx[r] = max(s_max[4 * R + r], 1);
        for (int64_t e = threadIdx.x; e < m; e += blockDim.x) {
            const int64_t p = p0 + e / kIt;
            double v[4];
            slice_load<NB>(a, p, R, c, v);
            uint32_t d[2 * kPairs][4];  // bf16 bits of digit d of row r
            bool some = false;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint64_t u = (uint64_t)__double_as_longlong(v[r]);
                const int ef = (int)(u >> 52) & 0x7ff;
                // |v| = M 2^(max(ef, 1) - 1075); F = v 2^(89 - e), 2^e the scale: M << (36 - s)
                int64_t M = (int64_t)(u & 0xfffffffffffffull) | (ef ? 0x10000000000000ll : 0ll);
                const int s = mx[r] - max(ef, 1);
                if (M != 0) {
                    some = true;
                    any |= 1 << r;
                    if (s >= kDeepBits) deep |= 1 << r;
                }
                if ((int64_t)u < 0) M = -M;
                int64_t H, L;  // F = 2^36 H + L, 0 <= L < 2^36
                if (s <= 36) {
                    H = M >> s;
                    L = (int64_t)((uint64_t)M << (36 - s) & 0xfffffffffull);
                } else {
                    const int w = min(s - 36, 62);
                    const int64_t F = (M + (1ll << (w - 1))) >> w;
                    H = F >> 36;
                    L = F & 0xfffffffffll;
                }
                L += 256ll * (1 + 512 + 512 * 512 + 512ll * 512 * 512);
                H += (L >> 36) + 256ll * (1 + 512 + 512 * 512 + 512ll * 512 * 512 + 512ll * 512 * 512 * 512);
#pragma unroll
                for (int k = 0; k < 4; ++k) d[9 - k][r] = digit_bf16((uint32_t)(L >> (9 * k)) & 511u);
#pragma unroll
                for (int k = 0; k < 5; ++k) d[5 - k][r] = digit_bf16((uint32_t)(H >> (9 * k)) & 511u);
                d[0][r] = digit_bf16((uint32_t)((int)(H >> 45) + 256));
            }
            const int64_t unit = NB * NB * p + NB * R + c / 4;
            // the unit's four columns are four neighbouring lanes
            const unsigned cols = __ballot_sync(0xfu << (threadIdx.x & 28), some);
            if ((c & 3) == 0) a.any[unit] = cols != 0;
#pragma unroll
            for (int t = 0; t < kPairs; ++t) {
                uint4 *o = t < 4 ? a.out + 16 * unit + 4 * t : a.tail + 4 * unit;
                o[c & 3] = make_uint4(d[2 * t][0] | d[2 * t][1] << 16, d[2 * t][2] | d[2 * t][3] << 16,
                                      d[2 * t + 1][0] | d[2 * t + 1][1] << 16, d[2 * t + 1][2] | d[2 * t + 1][3] << 16);
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (deep >> r & 1) s_deep[4 * R + r] = 1;
            if (any >> r & 1) s_any[4 * R + r] = 1;
        }
        __syncthreads();
        if (threadIdx.x < 4 * NB) {
            const int r = threadIdx.x, x = s_max[r];
            // v < 2^(ef - 1022)
            a.info[(int64_t)4 * NB * i + r] = (max(x, 1) - 1022 + kExpBias) | (s_deep[r] ? kDeep : 0) | (x == 0x7ff ? kBad : 0) |
                                            (s_any[r] ? 0 : kNone);
        }
        __syncthreads();
    }
}

// ---- the product -----------------------------------------------------------------------------
struct SlArgs {
    int n, b;
    const int32_t *order, *cta_first, *tile_nk, *tile_j, *tile_i0, *cpos, *cta_stages;
    const int64_t *cta_rec;
    const int32_t *pos;
    const char *As, *Xs;       // sliced units of op(A) and of X = op(B)^T: pairs 0-3
    const char *At, *Xt;       // and pair 4
    const int *Ai, *Xi;        // their row information
    double *C;
    const int64_t *c_tm;       // transpose map of C's pattern: also write C_ji = C_ij^T (or null)
    double alpha, beta;
    int *count;                // units left to k_listed: their number, ((row, sub-row, sub-column), block)
    int2 *list;
    int *err;
    unsigned long long wait_ns;
};

// Instruction descriptor of kind::f16 with bf16 operands, float32 accumulator, A and B MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16_mn(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// T 2^(x - kScaleBits) rounded to the nearest float64 (ties to even); *bits receives the length of |T|.
// |T| < 2^127.  Integer arithmetic: the FP64 pipe would take 20 times as long.  Results outside the
// normal range go through ldexp.
__device__ __forceinline__ double round_sum(__int128 T, int x, int *bits) {
    const bool neg = T < 0;
    const unsigned __int128 a = neg ? -(unsigned __int128)T : (unsigned __int128)T;
    const uint64_t h = (uint64_t)(a >> 64), l = (uint64_t)a;
    if (h == 0 && l == 0) {
        *bits = 0;
        return 0.0;
    }
    // 64 bits from the leading one: |T| = (m + rest 2^-64) 2^z
    const int c = __clzll((long long)(h ? h : l));
    const uint64_t rest = h ? l << c : 0;
    uint64_t m = h ? (c ? h << c | l >> (64 - c) : h) : l << c;
    const int z = (h ? 64 : 0) - c;
    *bits = 64 + z;
    const uint32_t tail = (uint32_t)m & 0x7ffu;
    m >>= 11;  // 53 bits
    m += (tail > 0x400u || (tail == 0x400u && (rest != 0 || (m & 1)))) ? 1 : 0;
    const int e = z + 63 - kScaleBits + x;  // 1.f 2^e
    if (e < -1021 || e > 1021) {
        const double d = ldexp((double)m, e - 52);
        return neg ? -d : d;
    }
    // m includes the leading bit, which adds one to the exponent field
    const uint64_t b = ((uint64_t)(e + 1022) << 52) + m;
    return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}

constexpr float kMagic = 12582912.f;      // 1.5 2^23: adding it to an integer rounds nothing up to 2^22
constexpr uint32_t kMagicBits = 0x4b400000;

template <int NB>
__global__ void __launch_bounds__(kThreads, 1) k_sl_product(SlArgs p) {
    constexpr int kRecN = kRec / (NB * NB);  // entries of a record
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kStages * kStageBytes + kRingBytes);
    // bars: full[kStages], empty[kStages], tfull[kBufs], upper parts free[kBufs], lower part free, drain
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStages + 2 * kBufs + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto empty = [&](int s) { return bar0 + 8u * (kStages + s); };
    auto tfull = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
    auto ufree = [&](int b) { return bar0 + 8u * (2 * kStages + kBufs + b); };
    const uint32_t lfree = bar0 + 8u * (2 * kStages + 2 * kBufs), drain = lfree + 8u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q0 = p.cta_first[blockIdx.x], q1 = p.cta_first[blockIdx.x + 1];

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full(s), 32 * kCopyWarps);  // per thread: its copies have landed
            mbar_init(empty(s), 1);
        }
        for (int b = 0; b < kBufs; ++b) {
            mbar_init(tfull(b), 1);
            mbar_init(ufree(b), kEpiWarps);
        }
        mbar_init(lfree, kEpiWarps);
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
        // ---- copies.  Warp w fills rows 8w .. 8w + 7 of every stage of 8 atoms k (warps 0 and 1 the
        // atoms j, warp 2 the atoms i).  One instruction moves pairs 0-3 of two blocks, a row's pair of
        // atoms k: lane l copies chunk (pair t = l / 8, column kk = l % 4) of block (l / 4) % 2, so that
        // eight lanes fill one core matrix (128 bytes, no bank conflicts).  A fifth instruction moves
        // pair 4 of a row's eight blocks.
        const int S = 2 * p.cta_stages[blockIdx.x];
        const int t = lane >> 3, par = (lane >> 2) & 1, kk = lane & 3;
        // The records come from HBM once each, so they are copied into a ring in shared memory
        // kRecAhead stages ahead (a wait on empty(slot) below means that the copies of three stages
        // back, and the record copies before them, have landed).  A lane needs the four atoms k of
        // its parity in each row: entries 4 par .. 4 par + 3.
        constexpr int kWarpRec = NB == 1 ? 64 : 4;  // entries of a record that a warp needs
        const int32_t *rec = p.pos + p.cta_rec[blockIdx.x] + kWarpRec * warp;
        const uint32_t ring = sbase + kStages * kStageBytes + 4 * kWarpRec * warp;
        auto fetch = [&](int st) {
            if (st < S && lane < kWarpRec / 4)
                cp_async16(ring + (uint32_t)(st % kRecRing) * (4 * kRecN) + 16 * lane, rec + (int64_t)kRecN * st + 4 * lane);
        };
        for (int st = 0; st < kRecAhead; ++st) fetch(st);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        // a core matrix of pair tt, pair kp of atoms k and row r lies at tt tstride + kp kstride + r kCore
        auto run = [&](const char *head, const char *tail, uint32_t dst0, auto tstride, auto kstride) {
            constexpr uint32_t ts = decltype(tstride)::value, ks = decltype(kstride)::value;
            const uint32_t in_core = (uint32_t)(64 * par + 16 * kk);
            head += 64 * t + 16 * kk + (NB == 1 ? 0 : kHead * par);
            tail += 16 * kk + (NB == 1 ? 0 : kTail * (2 * (t & 1) + par));  // this lane's pair of k is t
            for (int st = 0; st < S; ++st) {
                const int slot = st % kStages;
                bool ok = mbar_wait(empty(slot), ((uint32_t)(st / kStages) & 1u) ^ 1u, abort_flag, p.err, 1, p.wait_ns);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                const uint32_t base = sbase + (uint32_t)slot * kStageBytes + dst0 + in_core;
                const uint32_t from = ring + (uint32_t)(st % kRecRing) * (4 * kRecN);
                fetch(st + kRecAhead);
#pragma unroll
                for (int rr = 0; rr < 8; ++rr) {
                    const uint32_t dh = base + t * ts + rr * kCore, dt = base + 4 * ts + t * ks + rr * kCore;
                    if constexpr (NB == 1) {
                        int v[4], vt;
                        asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                                     : "r"(from + 16 * par + 32 * rr)
                                     : "memory");
                        asm volatile("ld.shared.s32 %0, [%1];" : "=r"(vt) : "r"(from + 16 * par + 32 * rr + 4 * t) : "memory");
#pragma unroll
                        for (int kp = 0; kp < kKP; ++kp) cp_async16_or_zero(dh + kp * ks, head, v[kp], kHead);
                        cp_async16_or_zero(dt, tail, vt, kTail);
                    } else {
                        // rows 0-3 and 4-7 are the sub-rows of an atom each, the stage's eight k the
                        // sub-columns of two atoms
                        int v[2];
                        asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(from + 8 * (rr >> 2)) : "memory");
#pragma unroll
                        for (int kp = 0; kp < kKP; ++kp)
                            cp_async16_or_zero(dh + kp * ks, head + kHead * (NB * (rr & 3) + 2 * (kp & 1)), v[kp >> 1], NB * NB * kHead);
                        cp_async16_or_zero(dt, tail + kTail * NB * (rr & 3), t < 2 ? v[0] : v[1], NB * NB * kTail);
                    }
                }
                cp_async_arrive(full(slot));
            }
        };
        if (warp < 2)
            run(p.Xs, p.Xt, (uint32_t)(8 * warp * kCore), std::integral_constant<int, kKP * kJT * kCore>(),
                std::integral_constant<int, kJT * kCore>());
        else
            run(p.As, p.At, (uint32_t)kPanelX, std::integral_constant<int, kG * kCore>(),
                std::integral_constant<int, kPairs * kG * kCore>());
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            // ---- MMAs: two stages (16 atoms k) to an accumulator, then a fresh one, so that no
            // sum passes 2^24.  Pair u of X times pairs b0 .. b0 + nb - 1 of A: columns from pair u + b0 on.
            int it = 0, st = 0;
            bool ok = true;
            int nk_n = q0 < q1 ? __ldg(p.tile_nk + __ldg(p.order + q0)) : 0;
            for (int q = q0; q < q1 && ok; ++q) {
                const int nk = nk_n;
                if (q + 1 < q1) nk_n = __ldg(p.tile_nk + __ldg(p.order + q + 1));
                for (int k0 = 0; k0 < nk && ok; k0 += kKS / NB, ++it, st += 2) {
                    const int buf = it % kBufs;
                    const uint32_t up = tmem + (uint32_t)(buf * kBufCols), low = tmem + (uint32_t)kLowAt;
                    auto part = [&](int h, bool lower) {
                        const uint32_t sx = sbase + (uint32_t)((st + h) % kStages) * kStageBytes, sa = sx + kPanelX;
#pragma unroll
                        for (int m = 0; m < kKP; m += 2)
#pragma unroll
                            for (int u = 0; u < kPairs; ++u) {
                                const int b0 = lower ? (u < kUpPairs ? kUpPairs - u : 0) : 0;
                                const int b1 = lower ? kPairs - u : kUpPairs - u;
                                if (b1 <= b0) continue;
                                const uint64_t bd = sdesc(sa + (m * kPairs + b0) * kG * kCore, kPairs * kG * kCore, kCore);
                                const uint64_t ad = sdesc(sx + (u * kKP + m) * kJT * kCore, kJT * kCore, kCore);
                                const uint32_t d = lower ? low + 64u * (u + b0 - kUpPairs) : up + 64u * u;
                                mma_bf16(d, ad, bd, idesc_bf16_mn(128, 64 * (b1 - b0)), (h > 0 || m > 0 || u > 0) ? 1u : 0u);
                            }
                    };
                    ok = mbar_wait(ufree(buf), ((uint32_t)(it / kBufs) & 1u) ^ 1u, abort_flag, p.err, 3, p.wait_ns);
                    for (int h = 0; h < 2 && ok; ++h) {
                        const int s2 = st + h;
                        ok = mbar_wait(full(s2 % kStages), (uint32_t)(s2 / kStages) & 1u, abort_flag, p.err, 2, p.wait_ns);
                        if (!ok) break;
                        fence_proxy_async();
                        tc_fence_after();
                        part(h, false);
                        if (h == 0) {
                            ok = mbar_wait(lfree, ((uint32_t)it & 1u) ^ 1u, abort_flag, p.err, 3, p.wait_ns);
                            if (!ok) break;
                            tc_fence_after();
                        }
                        part(h, true);
                        mma_commit(empty((st + h) % kStages));
                    }
                    if (!ok) break;
                    mma_commit(tfull(buf));
                }
            }
            mma_commit(drain);
            const unsigned long long t0 = globaltimer();
            while (!mbar_try(drain, 0u))
                if (globaltimer() - t0 > kWaitNs) {
                    atomicCAS(p.err, 0, 6);
                    break;
                }
        }
    } else if (warp >= kEpiWarp) {
        // ---- epilogue: lane m = 8 jj + 4 s + c of the accumulator (digit s of a pair of X); four
        // warps take the atoms i 0 and 1 of the group, four the next two, and so on (with 8 warps of
        // twice the work each, the latency of these chains showed).  Column 64 cp + 8 i +
        // 4 s' + r holds order s + o, o = 2 cp + s', as an integer of at most (cp + 1) 2^22.  Orders
        // 0 and 1 (cp = 0) turn into integers by adding 1.5 2^23 and taking the bits, the others by
        // conversion (a quarter of the rate, on a pipe of its own), and all are added to 64-bit
        // sums, so a result does not depend on how its terms are grouped.
        const int quad = warp & 3, i_lo = kEpiI * ((warp - kEpiWarp) >> 2);
        const int m = 32 * quad + lane;
        const int jj = m >> 3, s = (m >> 2) & 1, c = m & 3;
        const uint32_t tlane = tmem + ((uint32_t)(32 * quad) << 16) + 8u * i_lo;
        int it = 0;
        bool ok = true;
        // the next tile's numbers are read a tile ahead
        int t_n = 0, nk_n = 0, i0_n = 0, j_n = -1;
        auto look = [&](int q) {
            if (q >= q1) return;
            const int t = t_n = __ldg(p.order + q);
            nk_n = __ldg(p.tile_nk + t);
            i0_n = __ldg(p.tile_i0 + t);
            j_n = __ldg(p.tile_j + (int64_t)(kJT / NB) * t + jj / NB);
        };
        look(q0);
        for (int q = q0; q < q1 && ok; ++q) {
            const int t = t_n;
            const int ngr = nk_n / (kKS / NB), i0 = i0_n + i_lo / NB, j = j_n;
            look(q + 1);
            const int xi = j >= 0 ? p.Xi[4 * ((int64_t)NB * j + jj % NB) + c] : kBad;
            int cps[kEpiI];
#pragma unroll
            for (int i = 0; i < kEpiI; ++i) cps[i] = p.cpos[(int64_t)(128 / (NB * NB)) * t + (kJT / NB) * ((i_lo + i) / NB) + jj / NB];
            // per scalar of C: orders 0 to 3 in units of order 3 (and the magic constants' bits, which pass
            // 2^63 after 55 groups: unsigned, so that they wrap until the bias is taken off), orders 4
            // to 7 in units of order 7, orders 8 and 9 in units of order 9
            unsigned long long hi[kEpiI][4];
            long long mid[kEpiI][4], lo[kEpiI][4];
#pragma unroll
            for (int i = 0; i < kEpiI; ++i)
#pragma unroll
                for (int r = 0; r < 4; ++r) hi[i][r] = 0, mid[i][r] = lo[i][r] = 0;
            for (int gr = 0; gr < ngr; ++gr, ++it) {
                const int buf = it % kBufs;
                ok = mbar_wait(tfull(buf), (uint32_t)(it / kBufs) & 1u, abort_flag, p.err, 4, p.wait_ns);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                auto n = [](uint32_t v) { return (long long)__float2int_rn(__uint_as_float(v)); };
                auto mg = [](uint32_t v) { return (unsigned long long)__float_as_uint(__uint_as_float(v) + kMagic); };
                {
                    uint32_t w[kEpiI][2][8];  // orders 6 and 7, 8 and 9
#pragma unroll
                    for (int i = 0; i < kEpiI; ++i)
#pragma unroll
                        for (int k = 0; k < 2; ++k) tmem_ld8(tlane + (uint32_t)(kLowAt + 64 * k + 8 * i), w[i][k]);
                    tmem_wait_ld();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(lfree);
#pragma unroll
                    for (int i = 0; i < kEpiI; ++i)
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            mid[i][r] += n(w[i][0][r]) * (1 << 9);
                            mid[i][r] += n(w[i][0][4 + r]);
                            lo[i][r] += n(w[i][1][r]) * (1 << 9);
                            lo[i][r] += n(w[i][1][4 + r]);
                        }
                }
#pragma unroll
                for (int i = 0; i < kEpiI; ++i) {
                    uint32_t w[kUpPairs][8];
#pragma unroll
                    for (int k = 0; k < kUpPairs; ++k) tmem_ld8(tlane + (uint32_t)(buf * kBufCols + 64 * k + 8 * i), w[k]);
                    tmem_wait_ld();
                    if (i == kEpiI - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(ufree(buf));
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        hi[i][r] += mg(w[0][r]) * (1u << 27);
                        hi[i][r] += mg(w[0][4 + r]) * (1u << 18);
                        hi[i][r] += (unsigned long long)(n(w[1][r]) * (1 << 9));
                        hi[i][r] += (unsigned long long)n(w[1][4 + r]);
                        mid[i][r] += n(w[2][r]) * (1 << 27);
                        mid[i][r] += n(w[2][4 + r]) * (1 << 18);
                    }
                }
            }
            if (!ok) break;
            // sums of the two digits of a pair are in lanes l and l + 4: lane s = 0 finishes rows 0
            // and 1 of each block, lane s = 1 rows 2 and 3
            const unsigned long long bias = (unsigned long long)ngr * kMagicBits * ((1 << 27) + (1 << 18));  // of the magic constants
            const int least = kLeastBits + (32 - __clz(64 * ngr)) / 2;
            int ais[kEpiI][2];
#pragma unroll
            for (int i = 0; i < kEpiI; ++i)
#pragma unroll
                for (int u = 0; u < 2; ++u) ais[i][u] = p.Ai[4 * ((int64_t)NB * min(i0 + i / NB, p.n - 1) + (i_lo + i) % NB) + 2 * s + u];
#pragma unroll
            for (int i = 0; i < kEpiI; ++i) {
                // (a block that no stored pair of blocks adds to is -2 - cp)
                const int cp = cps[i] < -1 ? -2 - cps[i] : cps[i];
                const int ia = min(i0 + i / NB, p.n - 1);
                double w[2];
                int flags = xi & kBad;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    // a lane's sum in units of order 9, below 2^116 in size; the one of lane s = 0 counts
                    // 512-fold.  128 bits: hi 2^54 and mid 2^18 pass 64 after a few groups
                    auto sum = [&](int r) {
                        return (__int128)(long long)(hi[i][r] - bias) * (1ll << 54) + (__int128)mid[i][r] * (1 << 18) + lo[i][r];
                    };
                    const __int128 v0 = sum(u), v1 = sum(2 + u), give = s ? v0 : v1;
                    const uint64_t gl = __shfl_xor_sync(0xffffffffu, (unsigned long long)give, 4);
                    const long long gh = __shfl_xor_sync(0xffffffffu, (long long)(give >> 64), 4);
                    const __int128 got = (__int128)((unsigned __int128)(unsigned long long)gh << 64 | gl);
                    const __int128 T = s ? got * 512 + v1 : v0 * 512 + got;
                    const int ai = ais[i][u];
                    int bits;
                    w[u] = round_sum(T, (ai & 0xffff) + (xi & 0xffff) - 2 * kExpBias, &bits);
                    const int rows = ai | xi;
                    flags |= (rows & kBad) | (bits < least && (rows & (kDeep | kNone)) == kDeep ? kDeep : 0);
                }
                // any of the block's 16 sums: lanes c and s
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) flags |= __shfl_xor_sync(0xffffffffu, flags, o);
                if (cp < 0) continue;
                const int ld = NB == 1 ? 4 : p.b;
                const int Ri = (i_lo + i) % NB, Rj = jj % NB;
                if (NB > 1 && (4 * Ri >= ld || 4 * Rj >= ld)) continue;
                if (flags && cps[i] >= 0) {
                    if ((lane & 7) == 0) p.list[atomicAdd(p.count, 1)] = make_int2((ia * NB + Ri) * NB + Rj, cp);
                    continue;
                }
                const int row = 4 * Ri + 2 * s, col = 4 * Rj + c;
                if (cps[i] < 0) w[0] = w[1] = 0.0;  // also where zeros met digits of an infinity
                double *dst = p.C + (int64_t)(ld * ld) * cp + row * ld + col;
                const int64_t qc = p.c_tm ? p.c_tm[cp] : cp;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (NB > 1 && (row + u >= ld || col >= ld)) continue;
                    if (p.alpha != 1.0) w[u] *= p.alpha;
                    if (p.beta != 0.0) w[u] = fma(p.beta, dst[ld * u], w[u]);
                    dst[ld * u] = w[u];
                    if (NB > 1 && qc != cp) p.C[(int64_t)(ld * ld) * qc + col * ld + row + u] = w[u];
                }
                if (NB == 1 && qc != cp) *reinterpret_cast<double2 *>(p.C + 16 * qc + 4 * c + 2 * s) = make_double2(w[0], w[1]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

}  // namespace

int sliced_choice(lsq_geom g, int b, int ra, int rb, int rc, int upper, TcPlan **plan, bool *use, cudaStream_t s) {
    *use = false;
    const int nb = slice_units(b);
    if (nb == 0 || g_fma_products || g_group_rec || g->n == 0 || std::getenv("LSQ_PLAN_VARIANT")) return LSQ_OK;
    // LSQ_F64_SLICED fixes the choice (0 FMA, 1 slices), for tests
    const char *fixed = std::getenv("LSQ_F64_SLICED");
    if (fixed && std::atoi(fixed) == 0) return LSQ_OK;
    // the slices take 2.5 (4 x 4) to 8 (9 x 9) times their operands' memory, held as long as g: at most an
    // eighth of the device's, and a call that cannot have that much runs on FMA (whose plan they save: LS.L
    // of 2744 atoms holds 2.2 GB afterwards, 1.5 on FMA, the gradient of 1728 atoms 5.2 and 4.9)
    if ((size_t)kUnit * nb * nb * (size_t)(g->pats[ra].nnzb + g->pats[rb].nnzb) > g->mem_total / 8) return LSQ_OK;
    // The FMA schedules take 0.12 ns a triple of 4 x 4 blocks; the slices 9 to 11 ps a dense triple (a
    // third to a tenth of which are stored ones) and 3 us for their extra launches.  Measured, FMA
    // against slices, stored triples: 64 atoms, 153 k, 34.5 and 29.0 us; 216 atoms, 279 k, 50 and 59
    // us; 1.56 M, 196 and 106 us; 512 atoms, 101 k, 23 and 49 us; 660 k, 101 and 93 us; 1000 atoms,
    // 3.9 M, 467 and 469 us; 38 M, 4116 and 1189 us; 64 atoms of 13 x 13 blocks, 832, 32 and 28
    // us; 13 k, 111 and 74 us; 119 k, 801 and 165 us.  Larger blocks count by their scalars, b^3 against (4 nb)^3.
    const double per_triple = 15.0 * b * b * b / 64, per_dense = 1.4 * nb * nb * nb, launches = 375000.0;
    TcRule rule;
    // (a product has at least as many dense triples as stored ones)
    rule.can = [=](double n) { return n * (per_triple - per_dense) > launches; };
    rule.pays = [=](const TcPlan &p) {
        return p.max_nk <= kKS / nb * kMaxGroups && p.triples * per_triple > p.dense_triples * per_dense + launches;
    };
    return tensor_choice(g, ra, rb, rc, upper, tc_tile(0, nb), fixed != nullptr, rule, plan, use, s);
}

int sliced_block_matmul(lsq_geom g, int b, const TcPlan &pl, int ra, int ta, const double *A, int rb, int tb,
                        const double *B, int rc, double *C, double alpha, double beta, bool mirror, bool *done,
                        cudaStream_t s, bool b_sym, bool reuse_a) {
    const int nb = slice_units(b);
    LSQ_TRY(ensure_tmap(g, ra, s));
    LSQ_TRY(ensure_tmap(g, rb, s));
    if (pl.upper == 1 && mirror) LSQ_TRY(ensure_tmap(g, rc, s));
    SplitLock lock(g, s);
    LSQ_TRY(lock.status());
    *done = false;
    SplitSizes need;
    need.a = (size_t)kUnit * nb * nb * (size_t)std::max<int64_t>(g->pats[ra].nnzb, 1);
    need.x = (size_t)kUnit * nb * nb * (size_t)std::max<int64_t>(g->pats[rb].nnzb, 1);
    // (row information, then a byte for each unit)
    const size_t rows = 4 * (size_t)nb * g->n;
    auto info_bytes = [&](int r) { return sizeof(int) * rows + ((size_t)nb * nb * (size_t)g->pats[r].nnzb + 3) / 4 * 4; };
    need.ai = info_bytes(ra);
    need.xi = info_bytes(rb);
    need.list = sizeof(int) * (2 * (size_t)nb * nb * (size_t)std::max<int64_t>(g->pats[rc].nnzb, 1) + 2);
    SplitBuffers sb;
    const int got = lock.buffers(need, &sb);
    if (got == LSQ_ERR_OOM) {
        (void)cudaGetLastError();
        clear_error();
        return LSQ_OK;
    }
    LSQ_TRY(got);
    *done = true;
    int *err = nullptr;
    LSQ_TRY(dev_err_ptr(g, &err));
    SplitStore *st = lock.store();
    const bool keep = reuse_a && st && st->holds(A, ra, ta != 0, true);
    const int bmode = b_sym ? 2 : (tb == 0 ? 1 : 0);
    const int64_t ua = g->pats[ra].nnzb * nb * nb, ux = g->pats[rb].nnzb * nb * nb;
    SliceArgs sa, sx;
    sa.ptr = g->pats[ra].row_ptr.p;
    sa.tm = g->pats[ra].tmap.p;
    sa.X = A;
    sa.out = reinterpret_cast<uint4 *>(sb.a);
    sa.tail = sa.out + kHead / 16 * ua;
    sa.info = sb.ai;
    sa.any = reinterpret_cast<uint8_t *>(sb.ai + rows);
    sa.mode = ta ? 1 : 0;
    sa.b = sx.b = b;
    sx.ptr = g->pats[rb].row_ptr.p;
    sx.tm = g->pats[rb].tmap.p;
    sx.X = B;
    sx.out = reinterpret_cast<uint4 *>(sb.x);
    sx.tail = sx.out + kHead / 16 * ux;
    sx.info = sb.xi;
    sx.any = reinterpret_cast<uint8_t *>(sb.xi + rows);
    sx.mode = bmode;
    const int nops = keep ? 1 : 2;
    if (st) st->a_src = nullptr;
    note_launch();
    const int sgrid = std::max(1, std::min(g->n * nops, g->num_sms * 8));
    if (nb == 1) k_sl_slice<1><<<sgrid, 256, 0, s>>>(g->n, sx, sa, nops, sb.list);
    else k_sl_slice<4><<<sgrid, 1024, 0, s>>>(g->n, sx, sa, nops, sb.list);
    LSQ_CHECK_LAUNCH();
    if (st) st->set(A, ra, ta != 0, true);
    SlArgs a;
    a.n = g->n;
    a.order = pl.order.p;
    a.cta_first = pl.cta_first.p;
    a.b = b;
    a.tile_nk = pl.tile_nk.p;
    a.tile_j = pl.tile_j.p;
    a.tile_i0 = pl.tile_i0.p;
    a.cpos = pl.cpos.p;
    a.cta_stages = pl.cta_stages.p;
    a.cta_rec = pl.cta_rec.p;
    a.pos = pl.pos.p;
    a.As = sb.a;
    a.Xs = sb.x;
    a.At = a.As + kHead * ua;
    a.Xt = a.Xs + kHead * ux;
    a.Ai = sb.ai;
    a.Xi = sb.xi;
    a.C = C;
    a.c_tm = pl.upper == 1 && mirror ? g->pats[rc].tmap.p : nullptr;
    a.alpha = alpha;
    a.beta = beta;
    a.count = sb.list;
    a.list = reinterpret_cast<int2 *>(sb.list + 2);
    a.err = err;
    a.wait_ns = kWaitNs;
    if (const char *w = std::getenv("LSQ_TC_WAIT_NS")) a.wait_ns = std::strtoull(w, nullptr, 10);
    const auto product = nb == 1 ? k_sl_product<1> : k_sl_product<4>;
    LSQ_CUDA_TRY(cudaFuncSetAttribute(product, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes));
    note_launch();
    product<<<pl.grid, kThreads, kSmemBytes, s>>>(a);
    LSQ_CHECK_LAUNCH();
    LSQ_TRY(launch_listed(g, b, nb, ra, ta, A, rb, bmode, B, rc, C, alpha, beta, a.c_tm, a.count, a.list, s,
                          {sa.any, sx.any, sb.ai, sb.xi, nullptr, nullptr}));
    return lock.release();
}

}  // namespace lsq

// Blocks that a product on the tensor cores leaves to FMA: its epilogue lists them, and k_listed sums
// them as the FMA kernels would (shared by tc.cu and sliced.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lsq_internal.h"
#include "tc_ptx.h"

namespace lsq {
namespace {

// What is known of op(A) and X: a byte for each 4 x 4 unit, 0 if it is all zeros, and where infinities and
// NaN are (a zero times one counts): a word per scalar row with kBadRow set, or one word for all.
struct ListedFlags {
    const uint8_t *a_any, *x_any;
    const int *a_info, *x_info;    // float64
    const unsigned *a_odd, *x_odd; // float32
};

template <typename T>
struct ListedArgs {
    const int64_t *a_ptr, *x_ptr, *a_tm, *x_tm, *c_tm;
    const int32_t *a_col, *x_col, *c_col;
    const T *A, *B;
    int b, ta, bmode;     // block size; op(A) read through a_tm; X: 0 B's rows, 1 through x_tm, 2 B + B^T
    T *C;
    T alpha, beta;
    const int *count;
    const int2 *list;
    ListedFlags flags;
};
constexpr int kBadRow = 1 << 17;

// A warp per listed unit of a block (i, j), two lanes per element: the lanes look 32 atoms k of the
// shorter of row i of A and row j of X up in the other, then the halves of the warp add every other
// product found, A_ik X_jk^T.  (A lane per k and a reduction of 16 sums took 10 times the FP64
// instructions, which bound this; half a warp per unit ran the halves in turn.)  SYM: X is B + B^T (a
// kernel of its own: an addition that is predicated off still takes its turn on the FP64 pipe).
// With every block listed (2744 atoms, 336 M triples) this takes 43.5 ms where the FMA schedules take
// 35.7; the gradient's products at 1728 atoms 80 and 74 ms.
template <typename T, int NB, bool SYM>
__global__ void __launch_bounds__(256) k_listed(ListedArgs<T> a) {
    const int lane = threadIdx.x & 31, el = lane & 15;
    const bool upper = lane >= 16;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const int count = *a.count;
    const int b = NB == 1 ? 4 : a.b, bb = b * b;
    for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < count; w += nw) {
        const int2 e = a.list[w];
        const int i = e.x / (NB * NB), j = a.c_col[e.y];
        const int row = 4 * (e.x / NB % NB) + (el >> 2), col = 4 * (e.x % NB) + (el & 3);
        const int r = min(row, b - 1), c = min(col, b - 1);
        // element (r, t) of A_ik and (c, t) of X_jk: t steps of sa and sx
        const int sa = a.ta ? b : 1, oa = a.ta ? r : b * r, sx = a.bmode == 1 ? b : 1, ox = a.bmode == 1 ? c : b * c;
        const int64_t a0 = a.a_ptr[i], a1 = a.a_ptr[i + 1], x0 = a.x_ptr[j], x1 = a.x_ptr[j + 1];
        const bool walk_a = a1 - a0 <= x1 - x0;
        T part[4] = {0, 0, 0, 0};  // (shorter sums round less)
        // pairs with a unit that is stored but zero are passed over: an L that starts from its diagonal is
        // mostly such blocks, and all sums that are zero for it are listed
        const int Ri = e.x / NB % NB, Rj = e.x % NB;
        bool skip;
        if constexpr (sizeof(T) == 8) {
            int bad = 0;
            for (int k = 0; k < 4; ++k)
                bad |= a.flags.a_info[4 * ((int64_t)NB * i + Ri) + k] | a.flags.x_info[4 * ((int64_t)NB * j + Rj) + k];
            skip = !(bad & kBadRow);
        } else {
            skip = (*a.flags.a_odd | *a.flags.x_odd) == 0;
        }
        const uint8_t *a_any = a.flags.a_any, *x_any = a.flags.x_any;
        auto zero = [&](const uint8_t *any, int64_t p, int R) {
            return NB == 1 ? any[p] == 0 : *reinterpret_cast<const uint32_t *>(any + NB * (NB * p + R)) == 0;
        };
        for (int64_t q0 = walk_a ? a0 : x0; q0 < (walk_a ? a1 : x1); q0 += 32) {
            const int64_t q = q0 + lane;
            int64_t f = -1;
            if (q < (walk_a ? a1 : x1) && !(skip && (walk_a ? zero(a_any, q, Ri) : zero(x_any, q, Rj))))
                f = walk_a ? find_col(a.x_col, x0, x1, a.a_col[q]) : find_col(a.a_col, a0, a1, a.x_col[q]);
            if (f >= 0 && skip && (walk_a ? zero(x_any, f, Rj) : zero(a_any, f, Ri))) f = -1;
            unsigned found = __ballot_sync(0xffffffffu, f >= 0);
            while (found) {
                const int k0 = __ffs(found) - 1;
                found &= found - 1;
                const int k1 = __ffs(found) - 1;  // -1: none left for the upper half
                found &= found - (found ? 1 : 0);
                const int k = upper ? k1 : k0;
                const int64_t g = __shfl_sync(0xffffffffu, f, k < 0 ? 0 : k);
                if (k >= 0) {
                    const int64_t pa = walk_a ? q0 + k : g, px = walk_a ? g : q0 + k;
                    const T *Ab = a.A + bb * (a.ta ? a.a_tm[pa] : pa) + oa;
                    const T *Xb = a.B + bb * (a.bmode == 1 ? a.x_tm[px] : px) + ox;
                    const T *Xt = SYM ? a.B + bb * a.x_tm[px] + c : nullptr;
                    auto add = [&](int t, T &p) { p = fma(Ab[sa * t], SYM ? Xb[t] + Xt[b * t] : Xb[sx * t], p); };
                    int t = 0;
                    for (; t + 4 <= b; t += 4)
#pragma unroll
                        for (int u = 0; u < 4; ++u) add(t + u, part[u]);
                    if (NB > 1)
#pragma unroll 1
                        for (; t < b; ++t) add(t, part[0]);
                }
            }
        }
        T v = (part[0] + part[1]) + (part[2] + part[3]);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        if (upper) continue;
        if (row >= b || col >= b) continue;
        T *dst = a.C + (int64_t)bb * e.y + b * r + c;
        v *= a.alpha;
        if (a.beta != 0) v = fma(a.beta, *dst, v);
        *dst = v;
        if (a.c_tm) {
            const int64_t q = a.c_tm[e.y];
            if (q != e.y) a.C[bb * q + b * c + r] = v;
        }
    }
}

// The listed units of C = alpha op(A) op(B) + beta C (bmode: as ListedArgs; c_tm null or C's transpose map).
template <typename T>
int launch_listed(lsq_geom g, int b, int nb, int ra, int ta, const T *A, int rb, int bmode, const T *B, int rc, T *C,
                  double alpha, double beta, const int64_t *c_tm, const int *count, const int2 *list, cudaStream_t s,
                  const ListedFlags &flags) {
    const Pattern &PA = g->pats[ra], &PX = g->pats[rb];
    ListedArgs<T> a;
    a.a_ptr = PA.row_ptr.p;
    a.a_col = PA.col.p;
    a.a_tm = PA.tmap.p;
    a.x_ptr = PX.row_ptr.p;
    a.x_col = PX.col.p;
    a.x_tm = PX.tmap.p;
    a.c_tm = c_tm;
    a.c_col = g->pats[rc].col.p;
    a.A = A;
    a.B = B;
    a.b = b;
    a.ta = ta;
    a.bmode = bmode;
    a.C = C;
    a.alpha = (T)alpha;
    a.beta = (T)beta;
    a.count = count;
    a.list = list;
    a.flags = flags;
    const auto kern = nb == 1 ? (bmode == 2 ? k_listed<T, 1, true> : k_listed<T, 1, false>)
                              : (bmode == 2 ? k_listed<T, 4, true> : k_listed<T, 4, false>);
    note_launch();
    kern<<<g->num_sms * 4, 256, 0, s>>>(a);
    LSQ_CHECK_LAUNCH();
    return LSQ_OK;
}

}  // namespace
}  // namespace lsq

// K5: near-zone product with the stored blocks plus the self term (eq. 2):
//   y_a = alpha_a c_a + sum over stored pairs (a, b) of N_ab c_b   (alpha of a's scatterer),
// N_ab = P_a G_{a-b} P_b^T for boxes within Chebyshev distance 1 (the self block
// without coincident dipoles).  Blocks are nb_a x nb_b column-major, so a warp's lanes
// (one per test row) read a column contiguously.  HBM-bound on the blocks.
#include <algorithm>

#include "ie_internal.h"

namespace ie {
namespace {

constexpr int kNearWarps = 8;

// One CTA per test box a and NR right-hand sides, so that the columns of a call read each
// block once; its 8 warps split the stored blocks of row a.  A warp takes whole blocks: lane l
// owns rows l, l + 32, ... (ROWS of them, na <= 32 ROWS); the block's source coefficients sit in
// the warp's part of shared memory.  Columns go in groups of G whose loads are all issued before
// the group's arithmetic, so each lane keeps G x ROWS independent reads in flight.  Per block
// the sums run in FP32 and are added to two-float per-warp totals, combined in FP64 (the highs,
// converted by all warps: a conversion takes as long as an FP64 addition; the lows' sum in FP32).
// Measured (shell32, 729 MB of blocks): 128 us = 5.7 TB/s (156 us with shuffled coefficients, 16
// columns in flight and FP64 totals); 8 scatterers, 64-row boxes, four columns: 497 us for 1.25
// GB (935 us with a pass over the blocks per column; in pairs of columns per CTA 552 us).
// Nblk holds the blocks; with box_cols, columns r >= box_cols[a] take Nbeyond's instead.
static_assert(2 * ((27 + kNearWarps - 1) / kNearWarps) <= kTotalTerms, "a warp's blocks, short and beyond");
template <int ROWS, int NR>
__global__ void __launch_bounds__(kNearWarps * 32, ROWS * NR <= 4 ? 3 : ROWS == 2 ? 2 : 1)
near_kernel(const int32_t *__restrict__ nb, const int64_t *__restrict__ off, int64_t n,
            const int32_t *__restrict__ start, const int32_t *__restrict__ src,
            const int64_t *__restrict__ boff, const float2 *__restrict__ Nblk, const float2 *__restrict__ Nbeyond,
            const int32_t *__restrict__ box_cols, const double *__restrict__ alpha_box,
            const float2 *__restrict__ c, float2 *__restrict__ y, int nrhs, int items, const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    constexpr int G = ROWS == 1 ? 16 : (ROWS == 2 ? 8 : 4);     // columns per load group
    constexpr int X = 32 * ROWS;
    __shared__ __align__(16) float2 xs[kNearWarps][NR][X];      // c_b of the warp's block; then lows
    __shared__ double2 part[kNearWarps][X];                     // the totals' highs (lows: in xs)
    const int groups = (nrhs + NR - 1) / NR;             // a box's columns run next to each other
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const int a = item / groups, r0 = (item - a * groups) * NR;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int na = nb[a];
        const int within = box_cols ? box_cols[a] - r0 : NR;        // columns of this CTA that take Nblk
        float2 hi[ROWS][NR], lo[ROWS][NR];
#pragma unroll
        for (int k = 0; k < ROWS; ++k)
#pragma unroll
            for (int r = 0; r < NR; ++r) hi[k][r] = lo[k][r] = make_float2(0.f, 0.f);
        // (hi, lo) += the product of one block with the columns in shared memory
        auto block = [&](const float2 *N, int nbb) {
            float2 p[ROWS][NR];
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
#pragma unroll
                for (int r = 0; r < NR; ++r) p[k][r] = make_float2(0.f, 0.f);
            for (int j0 = 0; j0 < nbb; j0 += G) {
                float2 v[G][ROWS];
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int k = 0; k < ROWS; ++k) {
                        const int i = lane + 32 * k, j = j0 + g;
                        v[g][k] = (i < na && j < nbb) ? __ldcs(N + (int64_t)j * na + i) : make_float2(0.f, 0.f);
                    }
#pragma unroll
                for (int g = 0; g < G; g += 2)
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        // two columns' coefficients, the same address in every lane (zero past nbb)
                        const float4 x = *reinterpret_cast<const float4 *>(&xs[warp][r][j0 + g]);
#pragma unroll
                        for (int k = 0; k < ROWS; ++k) {
                            p[k][r].x = fmaf(v[g][k].x, x.x, fmaf(-v[g][k].y, x.y, p[k][r].x));
                            p[k][r].y = fmaf(v[g][k].x, x.y, fmaf(v[g][k].y, x.x, p[k][r].y));
                            p[k][r].x = fmaf(v[g + 1][k].x, x.z, fmaf(-v[g + 1][k].y, x.w, p[k][r].x));
                            p[k][r].y = fmaf(v[g + 1][k].x, x.w, fmaf(v[g + 1][k].y, x.z, p[k][r].y));
                        }
                    }
            }
#pragma unroll
            for (int k = 0; k < ROWS; ++k)
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    two_float_add(hi[k][r].x, lo[k][r].x, p[k][r].x);
                    two_float_add(hi[k][r].y, lo[k][r].y, p[k][r].y);
                }
        };
        const int t1 = start[a + 1];
        int t = start[a] + warp, b = 0, nbb = 0;
        int64_t ob = 0, bo = 0;
        auto next = [&](int q) {                     // the next block's place, ahead of its turn
            if (q >= t1) return;
            b = src[q];
            bo = boff[q];
            nbb = nb[b];
            ob = off[b];
        };
        // this block's coefficients (columns within = 1: r < within, 0: the others) into shared memory
        auto stage = [&](int64_t o, int cnt, bool inside) {
            bool any = false;                        // some column of the others is not zero
            __syncwarp();
#pragma unroll
            for (int r = 0; r < NR; ++r)
#pragma unroll
                for (int k = 0; k < ROWS; ++k) {
                    const int j = lane + 32 * k;
                    float2 x = j < cnt && r0 + r < nrhs ? c[(int64_t)(r0 + r) * n + o + j] : make_float2(0.f, 0.f);
                    if ((r < within) != inside) {
                        any |= !(x.x == 0.f && x.y == 0.f);
                        x = make_float2(0.f, 0.f);
                    }
                    xs[warp][r][j] = x;
                }
            __syncwarp();
            return any;
        };
        next(t);
        for (; t < t1; t += kNearWarps) {
            const int cnt = nbb;
            const int64_t o = ob, at = bo;
            const bool beyond = stage(o, cnt, true);
            next(t + kNearWarps);
            if (within > 0) block(Nblk + at, cnt);
            if (__any_sync(0xffffffffu, beyond)) {
                stage(o, cnt, false);
                block(Nbeyond + at, cnt);
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            __syncthreads();            // the sums before have been read
#pragma unroll
            for (int k = 0; k < ROWS; ++k) {
                part[warp][lane + 32 * k] = make_double2(hi[k][r].x, hi[k][r].y);
                xs[warp][0][lane + 32 * k] = make_float2(low_of(hi[k][r].x, lo[k][r].x), low_of(hi[k][r].y, lo[k][r].y));
            }
            __syncthreads();
            if (r0 + r < nrhs)
                for (int i = threadIdx.x; i < na; i += blockDim.x) {
                    double sr = 0, si = 0;
                    float lr = 0.f, li = 0.f;           // the lows' own sums: 2^-24 of the totals
#pragma unroll
                    for (int w = 0; w < kNearWarps; ++w) {
                        sr += part[w][i].x, lr += xs[w][0][i].x;
                        si += part[w][i].y, li += xs[w][0][i].y;
                    }
                    sr = kTotalTerms * (sr + lr);
                    si = kTotalTerms * (si + li);
                    const int64_t at = (int64_t)(r0 + r) * n + off[a] + i;
                    const float2 x = c[at];
                    const double alpha = alpha_box[a];
                    y[at] = make_float2((float)(sr + alpha * x.x), (float)(si + alpha * x.y));
                }
        }
        if (item + (int)gridDim.x < items) __syncthreads();         // xs has been read
    }
}

template <int ROWS>
void launch_rows(const ie_plan p, const float2 *blocks, const int32_t *cols, const float2 *c, float2 *y, int nrhs,
                 cudaStream_t st, const int *gate, int most_ctas) {
#define IE_NEAR(NR)                                                                                                \
    do {                                                                                                           \
        const int items = p->nbox * ((nrhs + NR - 1) / NR);                                                        \
        near_kernel<ROWS, NR><<<(unsigned)std::min(items, most_ctas), kNearWarps * 32, 0, st>>>(                   \
            p->d_nb, p->d_off, p->n, p->d_near_start, p->d_near_src, p->d_near_boff, blocks, p->d_Nblk, cols,      \
            p->d_alpha_box, c, y, nrhs, items, gate);                                                              \
    } while (0)
    // four columns of 192-row boxes would not fit the static shared memory
    constexpr int most = ROWS > 2 ? 2 : 4;
    if (nrhs == 1)
        IE_NEAR(1);
    else if (nrhs == 2)
        IE_NEAR(2);
    else
        IE_NEAR(most);
#undef IE_NEAR
}

}  // namespace

ie_status launch_near(const ie_plan p, const float2 *c, float2 *y, int nrhs, cudaStream_t st, const int *gate,
                      bool shorter, int most_ctas) {
    const float2 *blocks = shorter ? p->d_Nshort : p->d_Nblk;
    const int32_t *cols = shorter ? p->d_box_cols : nullptr;
    if (p->max_nb <= 32)
        launch_rows<1>(p, blocks, cols, c, y, nrhs, st, gate, most_ctas);
    else if (p->max_nb <= 64)
        launch_rows<2>(p, blocks, cols, c, y, nrhs, st, gate, most_ctas);
    else
        launch_rows<6>(p, blocks, cols, c, y, nrhs, st, gate, most_ctas);
    IE_CK_LAUNCH();
    return IE_OK;
}

}  // namespace ie

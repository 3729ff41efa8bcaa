// K2 / K4: mapping to uniform basis functions (Alg. 1, x_b = P_b^T c_b) and inverse
// mapping (Alg. 3, r_b = P_b y_b); the 16-bit hi/lo split of the mapped vectors for
// the tensor-core translation; the plane-wave excitation (§5) tested with P.
//
// Layouts: c, r: [rhs][n] complex64 (box b's coefficients at off[b] .. off[b+1]);
// P: [n][192] complex64 (row off[b]+i is basis function i of box b);
// X, Y: [rhs][nbox][192] complex64.  All HBM-bound: one CTA per box and up to four columns.
#include <algorithm>

#include "ie_internal.h"

namespace ie {
namespace {

// x[u] = sum_i P[i][u] c[i]: 192 threads, one per dipole unknown u, for NR right-hand sides
// (P is read once for them).  FP32 products in runs of 16 whose P values are all in flight
// together, runs added to two-float totals.  4 columns of 8 scatterers (335 MB of P): 78 us,
// 204 us with P read per column and FP64 totals; shell32, one column: 41 us = 6.0 TB/s.
template <int NR>
__global__ void __launch_bounds__(kNU) aggregate_kernel(const float2 *__restrict__ P, const int32_t *__restrict__ nb,
                                                        const int64_t *__restrict__ off, int64_t n, int nbox,
                                                        const float2 *__restrict__ c, float2 *__restrict__ X, int nrhs,
                                                        const int *__restrict__ gate) {
    chain_next();
    if (gate && *gate == 0) return;
    __shared__ float2 cs[kNU + 16][NR];
    const int b = blockIdx.x, r0 = blockIdx.y * NR, u = threadIdx.x;
    const int nbb = nb[b];
    const int64_t ob = off[b];
#pragma unroll
    for (int r = 0; r < NR; ++r)
        for (int i = u; i < kNU + 16; i += kNU)
            cs[i][r] = i < nbb && r0 + r < nrhs ? c[(int64_t)(r0 + r) * n + ob + i] : make_float2(0.f, 0.f);
    __syncthreads();
    const float2 *Pb = P + ob * kNU + u;
    float2 hi[NR], lo[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) hi[r] = lo[r] = make_float2(0.f, 0.f);
    for (int i0 = 0; i0 < nbb; i0 += 16) {
        float2 v[16], p[NR];
#pragma unroll
        for (int t = 0; t < 16; ++t) v[t] = i0 + t < nbb ? Pb[(int64_t)(i0 + t) * kNU] : make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < NR; ++r) p[r] = make_float2(0.f, 0.f);
#pragma unroll
        for (int t = 0; t < 16; ++t)
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const float2 cv = cs[i0 + t][r];
                p[r].x = fmaf(v[t].x, cv.x, fmaf(-v[t].y, cv.y, p[r].x));
                p[r].y = fmaf(v[t].x, cv.y, fmaf(v[t].y, cv.x, p[r].y));
            }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            two_float_add(hi[r].x, lo[r].x, p[r].x);
            two_float_add(hi[r].y, lo[r].y, p[r].y);
        }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r)
        if (r0 + r < nrhs)
            X[((int64_t)(r0 + r) * nbox + b) * kNU + u] =
                make_float2(two_float_total(hi[r].x, lo[r].x), two_float_total(hi[r].y, lo[r].y));
}

__global__ void copy_kernel(const float4 *__restrict__ a, float4 *__restrict__ b, int64_t n4,
                            const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n4) b[i] = a[i];
}

// 16-bit hi/lo split of X for the tensor-core path.  Layout [hl][rhs][nbox][chunk][reim][32]:
// per column 384 values, K-chunk major (chunk = u / 32), re and im rows of a chunk adjacent, so
// one K-chunk of a column (both rows) is 128 contiguous bytes for the tensor-core gathers.
// FP16: the column is scaled by 2^-e so that max |x| < 2^14; e is stored.
// With a symmetry map, copy z holds the signed-permuted input x^Q[u] = +-x[U_Q(u)] at Xtc + z *
// (2 planes); the scale is the same for every copy.
//
// Bound by the writes (48 copies: 74 KB per column).  A CTA splits its column once, keeps the
// halves in shared memory and writes kSplitCopies copies with 16-byte stores: a thread gathers
// eight unknowns of one copy and writes their four lines (hi, lo of re, im).  920 boxes, 48
// copies: network product 763 -> 739 us (a CTA per copy with 2-byte stores took 43 us of it).
constexpr int kSplitCopies = 8;
static_assert(kNU / 8 * kSplitCopies == kNU, "one thread per eight unknowns of a copy");
static_assert(kSym % kSplitCopies == 0, "whole groups of copies");
template <bool FP16>
__device__ __forceinline__ void split_column(int b, const float2 *__restrict__ X, int nbox, int nrhs,
                                             uint16_t *__restrict__ Xtc, int32_t *__restrict__ Xexp,
                                             float *__restrict__ Xinf, const uint16_t *__restrict__ symmap) {
    __shared__ uint2 halves[kNU];           // (hi re, hi im), (lo re, lo im)
    const int r = blockIdx.y, u = threadIdx.x;
    const int64_t col = (int64_t)r * nbox + b;
    const float2 x = X[col * kNU + u];
    const bool write_exp = blockIdx.z == 0;
    float scale = 1.f;
    if (FP16) {
        __shared__ float red[8], red2[8];
        __shared__ float s_scale;
        float m = fmaxf(fabsf(x.x), fabsf(x.y));
        float m2 = fmaf(x.y, x.y, x.x * x.x);     // for max_u |x_u| (the networks' input norm)
        for (int o = 16; o; o >>= 1) {
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            m2 = fmaxf(m2, __shfl_xor_sync(0xffffffffu, m2, o));
        }
        if ((u & 31) == 0) red[u >> 5] = m, red2[u >> 5] = m2;
        __syncthreads();
        if (u == 0) {
            float mm = 0.f, mm2 = 0.f;
            for (int w = 0; w < kNU / 32; ++w) mm = fmaxf(mm, red[w]), mm2 = fmaxf(mm2, red2[w]);
            if (write_exp && Xinf) Xinf[col] = sqrtf(mm2);
            int e = 0;
            if (mm > 0.f) {
                frexpf(mm, &e);
                e -= 14;
            }
            if (write_exp) Xexp[col] = e;
            s_scale = ldexpf(1.f, -e);
        }
        __syncthreads();
        scale = s_scale;
    } else if (u == 0 && write_exp) {
        Xexp[col] = 0;
    }
    const float v[2] = {x.x * scale, x.y * scale};
    uint32_t hi[2], lo[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        if (FP16) {
            __half h = __float2half_rn(v[t]);
            hi[t] = __half_as_ushort(h);
            lo[t] = __half_as_ushort(__float2half_rn(v[t] - __half2float(h)));
        } else {
            __nv_bfloat16 h = __float2bfloat16_rn(v[t]);
            hi[t] = __bfloat16_as_ushort(h);
            lo[t] = __bfloat16_as_ushort(__float2bfloat16_rn(v[t] - __bfloat162float(h)));
        }
    }
    const int64_t plane = (int64_t)nrhs * nbox * 2 * kNU;
    if (!symmap) {                          // one copy: every thread writes its own unknown
        uint16_t *cre = Xtc + col * 2 * kNU + (u >> 5) * 64 + (u & 31);
        cre[0] = hi[0];
        cre[32] = hi[1];
        cre[plane] = lo[0];
        cre[plane + 32] = lo[1];
        return;
    }
    halves[u] = make_uint2(hi[0] | hi[1] << 16, lo[0] | lo[1] << 16);
    __syncthreads();
    const int sg = blockIdx.z * kSplitCopies + u / (kNU / 8), k = u % (kNU / 8);    // copy, eight unknowns
    const uint4 e = __ldg(reinterpret_cast<const uint4 *>(symmap + (size_t)sg * kNU) + k);
    const uint32_t w[4] = {e.x, e.y, e.z, e.w};
    uint2 h[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t from = w[i >> 1] >> (16 * (i & 1));
        h[i] = halves[from & 0xFF];
        const uint32_t neg = from & 0x100 ? 0x80008000u : 0u;        // the halves of -x are negated
        h[i].x ^= neg;
        h[i].y ^= neg;
    }
    uint16_t *out = Xtc + 2 * plane * sg + col * 2 * kNU + (k >> 2) * 64 + (k & 3) * 8;
    uint4 re[2], im[2];                     // hi, lo: low halves of a pair of words are re, high ones im
    re[0] = make_uint4(__byte_perm(h[0].x, h[1].x, 0x5410), __byte_perm(h[2].x, h[3].x, 0x5410),
                       __byte_perm(h[4].x, h[5].x, 0x5410), __byte_perm(h[6].x, h[7].x, 0x5410));
    im[0] = make_uint4(__byte_perm(h[0].x, h[1].x, 0x7632), __byte_perm(h[2].x, h[3].x, 0x7632),
                       __byte_perm(h[4].x, h[5].x, 0x7632), __byte_perm(h[6].x, h[7].x, 0x7632));
    re[1] = make_uint4(__byte_perm(h[0].y, h[1].y, 0x5410), __byte_perm(h[2].y, h[3].y, 0x5410),
                       __byte_perm(h[4].y, h[5].y, 0x5410), __byte_perm(h[6].y, h[7].y, 0x5410));
    im[1] = make_uint4(__byte_perm(h[0].y, h[1].y, 0x7632), __byte_perm(h[2].y, h[3].y, 0x7632),
                       __byte_perm(h[4].y, h[5].y, 0x7632), __byte_perm(h[6].y, h[7].y, 0x7632));
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        *reinterpret_cast<uint4 *>(out + t * plane) = re[t];
        *reinterpret_cast<uint4 *>(out + t * plane + 32) = im[t];
    }
}

template <bool FP16>
__global__ void __launch_bounds__(kNU)
split_kernel(const float2 *__restrict__ X, int nbox, int nrhs, uint16_t *__restrict__ Xtc, int32_t *__restrict__ Xexp,
             float *__restrict__ Xinf, const uint16_t *__restrict__ symmap, const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    for (int b = blockIdx.x; b < nbox; b += gridDim.x) {
        if (b != (int)blockIdx.x) __syncthreads();      // the column before has been read
        split_column<FP16>(b, X, nbox, nrhs, Xtc, Xexp, Xinf, symmap);
    }
}

// Sum of an entry's nslab <= kSlabs partial sums (FP64), their reads in flight together.
__device__ __forceinline__ float2 slab_sum(const float2 *__restrict__ Y, int nslab, size_t slab_stride) {
    float2 w[kSlabs];
#pragma unroll
    for (int s = 0; s < kSlabs; ++s) w[s] = s < nslab ? Y[s * slab_stride] : make_float2(0.f, 0.f);
    double sr = 0, si = 0;
#pragma unroll
    for (int s = 0; s < kSlabs; ++s) {
        sr += w[s].x;
        si += w[s].y;
    }
    return make_float2((float)sr, (float)si);
}

// A far product's slabs in the form it took (p->d_form): nslab as given, or the blocks' kSlabs.
// False where it took neither (gated off).
__device__ __forceinline__ bool form_slabs(const int *__restrict__ form, int &nslab) {
    const int conv = form[0], blocks = form[1];
    if (blocks) nslab = kSlabs;
    return conv || blocks;
}

// r[i] (+)= sum_u P[i][u] y[u], y = sum over slabs (FP64), for NR right-hand sides (P is read
// once for them).  A warp takes four basis rows at a time, lanes over u, all 24 reads of P in
// flight; FP32 products and a tree that halves the number of sums a lane carries at each step
// (4 rows x NR columns x re / im sums: 9 exchanges instead of 40 at NR = 1, 31 instead of 160
// at NR = 4).  The 4 columns of 8 scatterers: 93 us, 234 us with P read per column; shell32, one
// column: 45 us = 5.5 TB/s.
constexpr int kDisThreads = 128;
template <int NR>
__global__ void __launch_bounds__(kDisThreads) disaggregate_kernel(const float2 *__restrict__ P, const int32_t *__restrict__ nb,
                                                           const int64_t *__restrict__ off, int64_t n, int nbox,
                                                           const float2 *__restrict__ Yslab, int nslab,
                                                           size_t slab_stride, float2 *__restrict__ out, int accumulate,
                                                           int identity, int nrhs, const int *__restrict__ gate,
                                                           const int *__restrict__ form) {
    if (gate && *gate == 0) return;
    if (form && !form_slabs(form, nslab)) return;
    constexpr int kRows = 4, M = 2 * kRows * NR;
    __shared__ float2 ys[NR][kNU];
    const int b = blockIdx.x, r0 = blockIdx.y * NR;
    const int64_t ob = off[b];
    for (int t = threadIdx.x; t < NR * kNU; t += blockDim.x) {
        const int r = t / kNU, u = t - r * kNU;
        float2 v = make_float2(0.f, 0.f);
        if (r0 + r < nrhs) {
            const float2 *Y = Yslab + ((int64_t)(r0 + r) * nbox + b) * kNU + u;
            if (nslab == 1) {
                v = *Y;
            } else if (nslab == 2) {
                v = *Y;
                const float2 w = Y[slab_stride];
                v = make_float2((float)((double)v.x + w.x), (float)((double)v.y + w.y));
            } else {
                v = slab_sum(Y, nslab, slab_stride);
            }
        }
        ys[r][u] = v;
    }
    __syncthreads();
    if (identity) {
        for (int t = threadIdx.x; t < NR * kNU; t += blockDim.x) {
            const int r = t / kNU, u = t - r * kNU;
            if (r0 + r >= nrhs) continue;
            float2 *o = out + (int64_t)(r0 + r) * n + ob + u;
            float2 v = ys[r][u];
            if (accumulate) {
                v.x += o->x;
                v.y += o->y;
            }
            *o = v;
        }
        return;
    }
    const int nbb = nb[b];
    const float2 *Pb = P + ob * kNU;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i0 = kRows * warp; i0 < nbb; i0 += kRows * nw) {
        float2 p[kRows][kNU / 32];
#pragma unroll
        for (int i = 0; i < kRows; ++i)
#pragma unroll
            for (int t = 0; t < kNU / 32; ++t)
                p[i][t] = i0 + i < nbb ? Pb[(int64_t)(i0 + i) * kNU + lane + 32 * t] : make_float2(0.f, 0.f);
        float v[M];                     // [row][column][re, im]
#pragma unroll
        for (int k = 0; k < M; ++k) v[k] = 0.f;
#pragma unroll
        for (int t = 0; t < kNU / 32; ++t)
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const float2 y = ys[r][lane + 32 * t];
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    float &re = v[2 * (i * NR + r)], &im = v[2 * (i * NR + r) + 1];
                    re = fmaf(p[i][t].x, y.x, fmaf(-p[i][t].y, y.y, re));
                    im = fmaf(p[i][t].x, y.y, fmaf(p[i][t].y, y.x, im));
                }
            }
        // after the step of bit o a lane keeps the sums whose index bit matches its own bit
        int idx = 0;
#pragma unroll
        for (int s = 0, o = 16, m = M; s < 5; ++s, o >>= 1) {
            if (m > 1) {
                m >>= 1;
                const bool up = lane & o;
#pragma unroll
                for (int k = 0; k < M / 2; ++k)
                    if (k < m) {
                        const float send = up ? v[k] : v[k + m], keep = up ? v[k + m] : v[k];
                        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                idx += up ? m : 0;
            } else {
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
            }
        }
        // lane holds sum idx; lanes that differ only below the last halving hold the same one
        constexpr int dup = 32 / M;
        const int i = idx / (2 * NR), r = idx / 2 % NR;
        if (lane % dup == 0 && i0 + i < nbb && r0 + r < nrhs) {
            float *o = reinterpret_cast<float *>(out + (int64_t)(r0 + r) * n + ob + i0 + i) + (idx & 1);
            *o = accumulate ? v[0] + *o : v[0];
        }
    }
}

__global__ void zero_kernel(float4 *__restrict__ p, int64_t n4, const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (; i < n4; i += stride) p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// nslab regions of n4 float4 each, stride4 float4 apart (blockIdx.y = region).
__global__ void zero_slabs_kernel(float4 *__restrict__ p, int64_t n4, int64_t stride4, const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    float4 *q = p + (int64_t)blockIdx.y * stride4;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x)
        q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void sum_slabs_kernel(const float2 *__restrict__ Yslab, int nslab, size_t slab_stride, int64_t count,
                                 float2 *__restrict__ Y, const int *__restrict__ form) {
    if (form && !form_slabs(form, nslab)) return;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    Y[i] = slab_sum(Yslab + i, nslab, slab_stride);
}

// Plane wave at the dipole sites, e[3s+a] = pol[a] exp(-j k khat . r_s) (FP64 phase),
// then v_b = P_b e_b as in disaggregate_kernel.
__global__ void plane_wave_kernel(double k, double a, int G, const int32_t *__restrict__ ijk,
                                  const float2 *__restrict__ P, const int32_t *__restrict__ nb,
                                  const int64_t *__restrict__ off, int64_t n,
                                  const double *__restrict__ khat, const double *__restrict__ pol,
                                  const int32_t *__restrict__ box_group, int nrhs,
                                  float2 *__restrict__ v, int identity) {
    __shared__ float2 es[kNU];
    int b = blockIdx.x, r = blockIdx.y;
    const int w = box_group[b] * nrhs + r;        // incidence of this scatterer's column r
    double h = a / kLattice;
    for (int s = threadIdx.x; s < kSites; s += blockDim.x) {
        int ii[3] = {s & 3, (s >> 2) & 3, s >> 4};
        double ph = 0;
        for (int c = 0; c < 3; ++c) {
            double pos = a * ((double)ijk[3 * b + c] + 0.5 - 0.5 * G) + h * (ii[c] + 0.5) - 0.5 * a;
            ph += khat[3 * w + c] * pos;
        }
        double sn, cs;
        sincos(-k * ph, &sn, &cs);
        for (int c = 0; c < 3; ++c) es[3 * s + c] = make_float2((float)(pol[3 * w + c] * cs), (float)(pol[3 * w + c] * sn));
    }
    __syncthreads();
    float2 *vb = v + (int64_t)r * n + off[b];
    if (identity) {
        for (int u = threadIdx.x; u < kNU; u += blockDim.x) vb[u] = es[u];
        return;
    }
    const float2 *Pb = P + off[b] * kNU;
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = warp; i < nb[b]; i += nw) {
        double pr = 0, pi = 0;
        const float2 *row = Pb + (int64_t)i * kNU;
        for (int t = 0; t < kNU / 32; ++t) {
            float2 p = row[lane + 32 * t];
            float2 e = es[lane + 32 * t];
            pr += (double)p.x * e.x - (double)p.y * e.y;
            pi += (double)p.x * e.y + (double)p.y * e.x;
        }
        for (int o = 16; o; o >>= 1) {
            pr += __shfl_xor_sync(0xffffffffu, pr, o);
            pi += __shfl_xor_sync(0xffffffffu, pi, o);
        }
        if (lane == 0) vb[i] = make_float2((float)pr, (float)pi);
    }
}

}  // namespace

ie_status launch_aggregate(const ie_plan p, const float2 *c, float2 *X, int nrhs, cudaStream_t st, const int *gate) {
    if (p->identity) {
        // n == nbox * 192 and [rhs][n] == [rhs][nbox][192]
        int64_t n4 = (int64_t)nrhs * p->n / 2;
        copy_kernel<<<(unsigned)((n4 + 255) / 256), 256, 0, st>>>(reinterpret_cast<const float4 *>(c),
                                                                  reinterpret_cast<float4 *>(X), n4, gate);
    } else {
#define IE_AGG(NR)                                                                                                 \
    aggregate_kernel<NR><<<dim3(p->nbox, (nrhs + NR - 1) / NR), kNU, 0, st>>>(p->d_P, p->d_nb, p->d_off, p->n, p->nbox, \
                                                                            c, X, nrhs, gate)
        if (nrhs == 1)
            IE_AGG(1);
        else if (nrhs == 2)
            IE_AGG(2);
        else
            IE_AGG(4);
#undef IE_AGG
    }
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_split_tc(const ie_plan p, const float2 *X, int nrhs, bool fp16, cudaStream_t st, const int *gate,
                          bool plain, int most_ctas) {
    const bool sym = p->sym && !plain;
    const int copies = sym ? kSym / kSplitCopies : 1;
    const dim3 grid(std::min(p->nbox, std::max(1, most_ctas / (nrhs * copies))), nrhs, copies);
    const uint16_t *map = sym ? p->d_symmap : nullptr;
    if (fp16)
        split_kernel<true><<<grid, kNU, 0, st>>>(X, p->nbox, nrhs, p->d_Xtc, p->d_Xexp, p->d_Xinf, map, gate);
    else
        split_kernel<false><<<grid, kNU, 0, st>>>(X, p->nbox, nrhs, p->d_Xtc, p->d_Xexp, nullptr, map, gate);
    IE_CK_LAUNCH();
    return IE_OK;
}

// The 48 signed-permuted copies x^Q[u] = +-x[U_Q(u)] of the FP32 translation input,
// layout [Q][rhs][nbox][192].
__global__ void permute_sym_kernel(const float2 *__restrict__ X, int nbox, int nrhs, const uint16_t *__restrict__ symmap,
                                   float2 *__restrict__ Xsym, const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    const int r = blockIdx.y, sg = blockIdx.z, u = threadIdx.x;
    const uint16_t e = symmap[sg * kNU + u];
    for (int b = blockIdx.x; b < nbox; b += gridDim.x) {
        const int64_t col = (int64_t)r * nbox + b;
        float2 x = X[col * kNU + (e & 0xFF)];
        if (e & 0x100) x = make_float2(-x.x, -x.y);
        Xsym[((int64_t)sg * nrhs * nbox + col) * kNU + u] = x;
    }
}

ie_status launch_permute_sym(const ie_plan p, const float2 *X, int nrhs, cudaStream_t st, const int *gate,
                             int most_ctas) {
    const dim3 grid(std::min(p->nbox, std::max(1, most_ctas / (nrhs * kSym))), nrhs, kSym);
    permute_sym_kernel<<<grid, kNU, 0, st>>>(X, p->nbox, nrhs, p->d_symmap, p->d_Xsym, gate);
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_disaggregate(const ie_plan p, const float2 *Yslab, int nslab, size_t stride, float2 *r, int nrhs,
                              bool accumulate, cudaStream_t st, const int *gate, const int *form) {
#define IE_DIS(NR)                                                                                                 \
    disaggregate_kernel<NR><<<dim3(p->nbox, (nrhs + NR - 1) / NR), kDisThreads, 0, st>>>(                          \
        p->d_P, p->d_nb, p->d_off, p->n, p->nbox, Yslab, nslab, stride, r, accumulate ? 1 : 0, p->identity ? 1 : 0, \
        nrhs, gate, form)
    if (nrhs == 1)
        IE_DIS(1);
    else if (nrhs == 2)
        IE_DIS(2);
    else
        IE_DIS(4);
#undef IE_DIS
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_zero(void *ptr, size_t bytes, cudaStream_t st, const int *gate) {
    if (bytes == 0) return IE_OK;
    if (bytes % 16) {
        set_error("launch_zero: size %zu not a multiple of 16", bytes);
        return IE_ERR_INVALID;
    }
    int64_t n4 = (int64_t)(bytes / 16);
    int64_t grid = (n4 + 255) / 256;
    if (grid > 4096) grid = 4096;
    zero_kernel<<<(unsigned)grid, 256, 0, st>>>(reinterpret_cast<float4 *>(ptr), n4, gate);
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_zero_slabs(float2 *base, int nslab, size_t stride, size_t count, cudaStream_t st, const int *gate,
                            int most_ctas) {
    if (count == 0 || nslab == 0) return IE_OK;
    if ((count * sizeof(float2)) % 16 || (stride * sizeof(float2)) % 16) {
        set_error("launch_zero_slabs: sizes not multiples of 16 bytes");
        return IE_ERR_INVALID;
    }
    const int64_t n4 = (int64_t)(count * sizeof(float2) / 16);
    int64_t gx = (n4 + 255) / 256;
    gx = std::min<int64_t>(gx, std::min(1024, std::max(1, most_ctas / nslab)));
    zero_slabs_kernel<<<dim3((unsigned)gx, (unsigned)nslab), 256, 0, st>>>(reinterpret_cast<float4 *>(base), n4,
                                                                          (int64_t)(stride * sizeof(float2) / 16),
                                                                          gate);
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_sum_slabs(const ie_plan p, const float2 *Yslab, int nslab, size_t stride, float2 *Y, int nrhs,
                           cudaStream_t st, const int *form) {
    int64_t count = (int64_t)nrhs * p->nbox * kNU;
    sum_slabs_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(Yslab, nslab, stride, count, Y, form);
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_plane_wave(const ie_plan p, const double *d_khat, const double *d_pol, int nrhs, float2 *v,
                            cudaStream_t st) {
    plane_wave_kernel<<<dim3(p->nbox, nrhs), 256, 0, st>>>(p->k, p->a, p->G, p->d_ijk, p->d_P, p->d_nb, p->d_off,
                                                           p->n, d_khat, d_pol, p->d_box_group, nrhs, v,
                                                           p->identity ? 1 : 0);
    IE_CK_LAUNCH();
    return IE_OK;
}

}  // namespace ie

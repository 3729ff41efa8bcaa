// K1: coupling blocks G_d (eq. 13) from the free-space dyadic Green's function
// (eq. 5, eq. 6), evaluated in FP64 on the device and stored for the translation
// kernels; and the stored near-zone blocks P_a G_{a-b} P_b^T (eq. 2).
//
// Geometry: dipole site s = ix + 4 iy + 16 iz of a box sits at the cell-centred
// offset h*((ix,iy,iz) + 1/2) - a/2 with h = a/4.  For test box = basis box + d the
// separation of test site l and basis site q is R = h (4 d + l - q), a multiple of
// the lattice spacing, so G_d depends only on d.
#include "ie_internal.h"

namespace ie {
namespace {

// One thread per (displacement, test site l, basis site q): the 3x3 block of G_d.
// row_major = false: layout [d][k][m] (k = basis unknown, m = test unknown), the
// FP32 translation kernel's A^T operand; true: [d][m][k].
__global__ void coupling_fp32_kernel(double k, double eta, double h, const int32_t *__restrict__ disp, int64_t nd,
                                     float2 *__restrict__ out, int row_major, int part) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nd * kSites * kSites) return;
    int64_t di = t / (kSites * kSites);
    int rem = (int)(t % (kSites * kSites));
    int q = rem / kSites;          // basis site (slower)
    int l = rem % kSites;          // test site (faster: coalesced m)
    int dx = disp[3 * di], dy = disp[3 * di + 1], dz = disp[3 * di + 2];
    int mx = 4 * dx + (l & 3) - (q & 3);
    int my = 4 * dy + ((l >> 2) & 3) - ((q >> 2) & 3);
    int mz = 4 * dz + (l >> 4) - (q >> 4);
    double2 D[9];
    const int reach = max(abs(mx), max(abs(my), abs(mz)));
    const bool skip = reach == 0 || (part == kShortSites && reach > kNearReach) ||
                            (part == kLongSitesNegated && reach <= kNearReach);
    const float sg = part == kLongSitesNegated ? -1.f : 1.f;
    if (!skip) dyad_fp64(k, eta, h * mx, h * my, h * mz, D);
    float2 *blk = out + di * (int64_t)kNU * kNU;
#pragma unroll
    for (int al = 0; al < 3; ++al)
#pragma unroll
        for (int be = 0; be < 3; ++be) {
            float2 v = skip ? make_float2(0.f, 0.f)
                                  : make_float2(sg * (float)D[3 * al + be].x, sg * (float)D[3 * al + be].y);
            int m = 3 * l + al, kk = 3 * q + be;
            if (row_major)
                blk[(int64_t)m * kNU + kk] = v;
            else
                blk[(int64_t)kk * kNU + m] = v;
        }
}

// Tensor-core images of every far coupling block, from the FP32 store.
// Real embedding of y = G x with G = Gr + j Gi, split operands x = [xr; xi]:
// real row 2m holds Gr[m][:], row 2m+1 holds Gi[m][:]; the GEMM against the
// columns xr and xi gives Gr xr, Gr xi, Gi xr, Gi xi, combined in the epilogue.
// Image (mb, kc, hl): rows 128 mb .. +127, source unknowns 32 kc .. +31, hi or lo
// 16-bit part, in the 64-byte-swizzled K-major layout of tcgen05.mma: row r is 64 B,
// its 16-byte chunk c lands at chunk c ^ ((r / 2) mod 4).  One CTA per displacement.
// fp16: scaled by 2^-e (e stored) so that |entries| <= 2^14.
template <bool FP16>
__global__ void coupling_tc_kernel(const float2 *__restrict__ Cs, int64_t nd, uint16_t *__restrict__ out,
                                   int32_t *__restrict__ exps) {
    int64_t di = blockIdx.x;
    if (di >= nd) return;
    const float2 *blk = Cs + di * (int64_t)kNU * kNU;   // [k][m]
    __shared__ float red[32];
    __shared__ float s_scale;
    float scale = 1.f;
    if (FP16) {
        float mx = 0.f;
        for (int i = threadIdx.x; i < kNU * kNU; i += blockDim.x) {
            float2 v = blk[i];
            mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
        }
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
        __syncthreads();
        if (threadIdx.x == 0) {
            float m = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
            int e = 0;
            if (m > 0.f) {
                frexpf(m, &e);     // m = f 2^e, f in [0.5, 1)
                e -= 14;           // m 2^-e < 2^14
            }
            exps[di] = e;
            s_scale = ldexpf(1.f, -e);
        }
        __syncthreads();
        scale = s_scale;
    }
    uint16_t *img0 = out + di * (int64_t)kTcDispElems;
    // 36 images x 128 rows x 4 chunks of 16 bytes
    for (int w = threadIdx.x; w < kTcImagesPerDisp * 128 * 4; w += blockDim.x) {
        int c = w & 3;
        int r = (w >> 2) & 127;
        int img = w >> 9;               // (mb * 6 + kc) * 2 + hl
        int hl = img & 1;
        int kc = (img >> 1) % kTcKChunks;
        int mb = (img >> 1) / kTcKChunks;
        int R = 128 * mb + r;
        int m = R >> 1, part = R & 1;
        uint16_t vals[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            int kk = kTcK * kc + 8 * c + e;
            float2 g = blk[(int64_t)kk * kNU + m];
            float x = (part ? g.y : g.x) * scale;
            if (FP16) {
                __half hi = __float2half_rn(x);
                __half lo = __float2half_rn(x - __half2float(hi));
                vals[e] = __half_as_ushort(hl ? lo : hi);
            } else {
                __nv_bfloat16 hi = __float2bfloat16_rn(x);
                __nv_bfloat16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
                vals[e] = __bfloat16_as_ushort(hl ? lo : hi);
            }
        }
        uint4 pk;
        pk.x = vals[0] | ((uint32_t)vals[1] << 16);
        pk.y = vals[2] | ((uint32_t)vals[3] << 16);
        pk.z = vals[4] | ((uint32_t)vals[5] << 16);
        pk.w = vals[6] | ((uint32_t)vals[7] << 16);
        uint4 *dst = reinterpret_cast<uint4 *>(img0 + (int64_t)img * kTcImageElems + r * kTcK +
                                               8 * (c ^ ((r >> 1) & 3)));
        *dst = pk;
    }
}

// Near blocks: N_ab = P_a G_{a-b} P_b^T (test box a, basis box b), nb_a x nb_b,
// column-major, and with Nshort the same from the blocks cut to kNearReach (Cnear + 27
// blocks).  One CTA per stored pair; basis columns in chunks of 32.  W = G P_b^T is a
// 192 x 32 register-tiled product (6 x 4 complex per thread, G chunks through shared memory,
// double-buffered), N = P_a W follows from shared memory.  Sums of 32 terms run in FP32,
// the chunks' sums are added as two-float pairs (an FP64 addition would take as long as the
// 32 multiply-adds before it).  FP32 rate bound: both block sets of the 32^3 shell in 52 ms
// (38 TFLOP/s; one set took 122 ms with a sum per thread and G read per term), the 16^3
// shell's in 13 ms (31).
constexpr int kNearJ = 32, kNearKC = 16, kNearThreads = 256;
struct SmemNear {
    float2 Pb[kNU][kNearJ];             // [k][j]
    union {
        float2 A[2][kNearKC][kNU];      // G chunk [k][m]
        float2 W[kNU][kNearJ];          // [m][j], once G has been read
    };
};
static_assert(sizeof(float2) * kNU * kNearJ == sizeof(float2) * 2 * kNearKC * kNU, "W overlays the chunks");

__global__ void __launch_bounds__(kNearThreads)
near_blocks_kernel(const float2 *__restrict__ Cnear,     // [27 or 54][k][m], index by e
                   const int32_t *__restrict__ ijk, const int32_t *__restrict__ nb, const int64_t *__restrict__ off,
                   const float2 *__restrict__ P, const int32_t *__restrict__ pair_a, const int32_t *__restrict__ pair_b,
                   const int64_t *__restrict__ boff, float2 *__restrict__ Nblk, float2 *__restrict__ Nshort) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmemNear &S = *reinterpret_cast<SmemNear *>(smem_raw);
    const int64_t pi = blockIdx.x;
    const int tid = threadIdx.x, a = pair_a[pi], b = pair_b[pi];
    const int ex = ijk[3 * a] - ijk[3 * b], ey = ijk[3 * a + 1] - ijk[3 * b + 1], ez = ijk[3 * a + 2] - ijk[3 * b + 2];
    const int e = (ex + 1) * 9 + (ey + 1) * 3 + (ez + 1);
    const int na = nb[a], nbb = nb[b], tm = tid >> 3, tn = tid & 7;   // rows 2 tm, + 1 (+ 64 j); columns 4 tn ..
    const float2 *Pa = P + off[a] * kNU, *Pbg = P + off[b] * kNU;
    for (int j0 = 0; j0 < nbb; j0 += kNearJ) {
        const int nj = min(kNearJ, nbb - j0);
        __syncthreads();
        for (int i = tid; i < kNearJ * kNU; i += kNearThreads) {
            const int jj = i / kNU, k = i - jj * kNU;
            S.Pb[k][jj] = jj < nj ? Pbg[(int64_t)(j0 + jj) * kNU + k] : make_float2(0.f, 0.f);
        }
        // the box's own block has no site pair beyond kNearReach: one product serves both
        for (int part = 0; part < (Nshort && e != 13 ? 2 : 1); ++part) {
            const float2 *C = Cnear + (int64_t)(e + 27 * part) * kNU * kNU;   // [k][m]
            float2 *N = (part ? Nshort : Nblk) + boff[pi];
            auto load = [&](int kc, int buf) {
                const float4 *g = reinterpret_cast<const float4 *>(C + (int64_t)kc * kNearKC * kNU);
                float4 *s = reinterpret_cast<float4 *>(&S.A[buf][0][0]);
#pragma unroll
                for (int t = 0; t < kNearKC * kNU / 2 / kNearThreads; ++t) {
                    const uint32_t d = (uint32_t)__cvta_generic_to_shared(s + tid + t * kNearThreads);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(g + tid + t * kNearThreads));
                }
                asm volatile("cp.async.commit_group;\n" ::);
            };
            float2 hi[6][4], lo[6][4], acc[6][4];
#pragma unroll
            for (int i = 0; i < 6; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) hi[i][j] = lo[i][j] = acc[i][j] = make_float2(0.f, 0.f);
            __syncthreads();        // W of the part before has been read
            load(0, 0);
            for (int kc = 0; kc < kNU / kNearKC; ++kc) {
                if (kc + 1 < kNU / kNearKC) {
                    load(kc + 1, (kc + 1) & 1);
                    asm volatile("cp.async.wait_group 1;\n" ::);
                } else {
                    asm volatile("cp.async.wait_group 0;\n" ::);
                }
                __syncthreads();
#pragma unroll 2
                for (int kk = 0; kk < kNearKC; ++kk) {
                    float2 g[6], p[4];
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const float4 v = *reinterpret_cast<const float4 *>(&S.A[kc & 1][kk][2 * tm + 64 * j]);
                        g[2 * j] = make_float2(v.x, v.y);
                        g[2 * j + 1] = make_float2(v.z, v.w);
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const float4 v = *reinterpret_cast<const float4 *>(&S.Pb[kc * kNearKC + kk][4 * tn + 2 * j]);
                        p[2 * j] = make_float2(v.x, v.y);
                        p[2 * j + 1] = make_float2(v.z, v.w);
                    }
#pragma unroll
                    for (int i = 0; i < 6; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            acc[i][j].x = fmaf(g[i].x, p[j].x, fmaf(-g[i].y, p[j].y, acc[i][j].x));
                            acc[i][j].y = fmaf(g[i].x, p[j].y, fmaf(g[i].y, p[j].x, acc[i][j].y));
                        }
                }
                if (kc & 1) {       // every 32 terms
#pragma unroll
                    for (int i = 0; i < 6; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            two_float_add(hi[i][j].x, lo[i][j].x, acc[i][j].x);
                            two_float_add(hi[i][j].y, lo[i][j].y, acc[i][j].y);
                            acc[i][j] = make_float2(0.f, 0.f);
                        }
                }
                __syncthreads();
            }
#pragma unroll
            for (int i = 0; i < 6; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    S.W[2 * tm + 64 * (i >> 1) + (i & 1)][4 * tn + j] =
                        make_float2(two_float_total(hi[i][j].x, lo[i][j].x),
                                    two_float_total(hi[i][j].y, lo[i][j].y));
            __syncthreads();
            // N[i][j0 + jj] = sum_m Pa[i][m] W[m][jj]: lane = column, a warp takes four rows at a time
            const int jj = tid & 31, warp = tid >> 5;
            for (int i0 = 4 * warp; i0 < na; i0 += 4 * (kNearThreads / 32)) {
                float2 h[4], l[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) h[r] = l[r] = make_float2(0.f, 0.f);
                for (int m0 = 0; m0 < kNU; m0 += 32) {
                    float2 q[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) q[r] = make_float2(0.f, 0.f);
#pragma unroll 4
                    for (int m = m0; m < m0 + 32; ++m) {
                        const float2 w = S.W[m][jj];
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float2 pa = __ldg(Pa + (int64_t)min(i0 + r, na - 1) * kNU + m);
                            q[r].x = fmaf(pa.x, w.x, fmaf(-pa.y, w.y, q[r].x));
                            q[r].y = fmaf(pa.x, w.y, fmaf(pa.y, w.x, q[r].y));
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        two_float_add(h[r].x, l[r].x, q[r].x);
                        two_float_add(h[r].y, l[r].y, q[r].y);
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (i0 + r < na && jj < nj) {
                        const float2 v =
                            make_float2(two_float_total(h[r].x, l[r].x), two_float_total(h[r].y, l[r].y));
                        N[(int64_t)(j0 + jj) * na + i0 + r] = v;
                        if (Nshort && e == 13) Nshort[boff[pi] + (int64_t)(j0 + jj) * na + i0 + r] = v;
                    }
            }
        }
    }
}

// Identity mapping: the near block is G_e itself (192 x 192, column-major = [k][m]).
__global__ void near_blocks_identity_kernel(const float2 *__restrict__ Cnear, const int32_t *__restrict__ ijk,
                                            const int32_t *__restrict__ pair_a, const int32_t *__restrict__ pair_b,
                                            const int64_t *__restrict__ boff, int64_t npairs,
                                            float2 *__restrict__ Nblk, float2 *__restrict__ Nshort) {
    int64_t pi = blockIdx.x;
    if (pi >= npairs) return;
    int a = pair_a[pi], b = pair_b[pi];
    int e = (ijk[3 * a] - ijk[3 * b] + 1) * 9 + (ijk[3 * a + 1] - ijk[3 * b + 1] + 1) * 3 +
            (ijk[3 * a + 2] - ijk[3 * b + 2] + 1);
    const float4 *src = reinterpret_cast<const float4 *>(Cnear + (int64_t)e * kNU * kNU);
    float4 *dst = reinterpret_cast<float4 *>(Nblk + boff[pi]);
    for (int i = threadIdx.x; i < kNU * kNU / 2; i += blockDim.x) dst[i] = src[i];
    if (!Nshort) return;
    src += (int64_t)27 * kNU * kNU / 2;
    dst = reinterpret_cast<float4 *>(Nshort + boff[pi]);
    for (int i = threadIdx.x; i < kNU * kNU / 2; i += blockDim.x) dst[i] = src[i];
}

}  // namespace

ie_status launch_coupling_fp32(double k, double eta, double a, const int32_t *d_disp, int64_t nd, float2 *out,
                               bool row_major, cudaStream_t st, BlockPart part) {
    if (nd <= 0) return IE_OK;
    int64_t threads = nd * kSites * kSites;
    int bs = 256;
    int64_t grid = (threads + bs - 1) / bs;
    coupling_fp32_kernel<<<(unsigned)grid, bs, 0, st>>>(k, eta, a / kLattice, d_disp, nd, out, row_major ? 1 : 0, part);
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_coupling_simt(const ie_plan p, const int32_t *d_disp, int64_t nd, float2 *out, bool row_major,
                               cudaStream_t st) {
    return launch_coupling_fp32(p->k, p->eta, p->a, d_disp, nd, out, row_major, st);
}

ie_status launch_coupling_tc(const float2 *Cs, int64_t nd, uint16_t *out, int32_t *exps, bool fp16, cudaStream_t st) {
    if (nd <= 0) return IE_OK;
    if (fp16)
        coupling_tc_kernel<true><<<(unsigned)nd, 256, 0, st>>>(Cs, nd, out, exps);
    else
        coupling_tc_kernel<false><<<(unsigned)nd, 256, 0, st>>>(Cs, nd, out, exps);
    IE_CK_LAUNCH();
    return IE_OK;
}

ie_status launch_near_blocks(ie_plan p, cudaStream_t st) {
    if (p->n_near_pairs == 0) return IE_OK;
    // the 27 near displacements, e = (ex+1)*9 + (ey+1)*3 + (ez+1)
    std::vector<int32_t> ds(27 * 3);
    for (int e = 0; e < 27; ++e) {
        ds[3 * e] = e / 9 - 1;
        ds[3 * e + 1] = (e / 3) % 3 - 1;
        ds[3 * e + 2] = e % 3 - 1;
    }
    int32_t *d_ds = nullptr;
    float2 *d_C = nullptr;
    int32_t *d_pa = nullptr;
    ie_status room = scratch_alloc(&d_ds, ds.size(), st);
    if (room == IE_OK) room = scratch_alloc(&d_C, (size_t)54 * kNU * kNU, st);
    if (room == IE_OK) room = scratch_alloc(&d_pa, (size_t)p->n_near_pairs, st);
    if (room != IE_OK) {
        for (void *q : {(void *)d_ds, (void *)d_C})
            if (q) cudaFreeAsync(q, st);
        return room;
    }
    IE_CK(cudaMemcpyAsync(d_ds, ds.data(), ds.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    IE_TRY(launch_coupling_simt(p, d_ds, 27, d_C, false, st));
    if (p->d_Nshort)
        IE_TRY(launch_coupling_fp32(p->k, p->eta, p->a, d_ds, 27, d_C + (size_t)27 * kNU * kNU, false, st, kShortSites));
    if (p->d_Cadj) {
        IE_TRY(launch_coupling_fp32(p->k, p->eta, p->a, d_ds, 27, p->d_Cadj, false, st, kLongSitesNegated));
        if (p->d_Cadj_bf16) IE_TRY(launch_coupling_tc(p->d_Cadj, 27, p->d_Cadj_bf16, nullptr, false, st));
        if (p->d_Cadj_fp16) IE_TRY(launch_coupling_tc(p->d_Cadj, 27, p->d_Cadj_fp16, p->d_Cadj_exp16, true, st));
    }
    // target box of every stored pair
    std::vector<int32_t> start(p->nbox + 1);
    IE_CK(cudaMemcpyAsync(start.data(), p->d_near_start, start.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    IE_CK(cudaStreamSynchronize(st));
    std::vector<int32_t> pa(p->n_near_pairs);
    for (int a = 0; a < p->nbox; ++a)
        for (int i = start[a]; i < start[a + 1]; ++i) pa[i] = a;
    IE_CK(cudaMemcpyAsync(d_pa, pa.data(), pa.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    if (p->identity) {
        near_blocks_identity_kernel<<<(unsigned)p->n_near_pairs, 256, 0, st>>>(d_C, p->d_ijk, d_pa, p->d_near_src,
                                                                               p->d_near_boff, p->n_near_pairs,
                                                                               p->d_Nblk, p->d_Nshort);
    } else {
        IE_CK(cudaFuncSetAttribute(near_blocks_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)sizeof(SmemNear)));
        near_blocks_kernel<<<(unsigned)p->n_near_pairs, kNearThreads, sizeof(SmemNear), st>>>(
            d_C, p->d_ijk, p->d_nb, p->d_off, p->d_P, d_pa, p->d_near_src, p->d_near_boff, p->d_Nblk, p->d_Nshort);
    }
    IE_CK_LAUNCH();
    IE_CK(cudaFreeAsync(d_ds, st));
    IE_CK(cudaFreeAsync(d_C, st));
    IE_CK(cudaFreeAsync(d_pa, st));
    return IE_OK;
}

}  // namespace ie

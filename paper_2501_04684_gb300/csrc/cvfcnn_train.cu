// Training of the CVFCNN translation networks (§3), first stage, on the GPU.
//
// One network per canonical displacement c = sorted |d| (192 -> H -> 192, complex,
// Cartesian ReLU on the hidden layer; the network is applied to x / ||x||_inf and its
// output is scaled back, so it learns G_c on the unit l-inf ball).  The paper's first
// training stage: inputs whose real and imaginary parts are uniform in [-1, 1]
// (normalised by their l-inf norm), the DGFA product G_c x as the target, mean square
// error, Adam; the stage ends when the relative l2 error of the outputs on a test set of
// the same distribution, e^u of eq. 171, is below the tolerance (1e-3 in the paper).
// The paper's second stage needs RWG-mapped surface data (absent here) and is not run.
//
// Layout: one CTA per network (persistent over networks), 256 threads; an Adam step
// sums the gradients of `minibatches` minibatches of 32 samples, each held in shared
// memory in turn:
//   X  [192][34]  inputs x / s (column j = sample j; rows of 272 bytes: 16-byte reads along
//                 a row and down the rows are free of bank conflicts)
//   R  [192][34]  target G x / (s g) (g = max |G| of the block, so the weights the
//                 optimiser sees are of order one), then the output residual
//   Z  [64][34]   hidden pre-activations, then the back-propagated hidden gradient
//   Hh [64][34]   hidden activations
//   A              two chunks of the matrix a product reads from global memory (cp.async)
// The six products of a minibatch run on register tiles: 6 x 4 outputs per thread for the
// 192-row ones (target, output layer), 4 x 2 for the 64-row ones (hidden layer, hidden
// gradient), 4 x 6 for the two weight gradients (a thread's rows in two halves).  FP32 rate bound, one CTA (two warps per
// scheduler) per SM: 192 x 192 + 5 x 192 H complex multiply-adds per sample, 0.17 ms per step
// of 128 samples at the peak rate for H = 50; 0.43 ms measured (1.0 ms with operands
// read per multiply-add from global memory and one gradient entry per thread at a time).
// Weights and Adam moments live in global memory (L2-resident while the CTA trains):
// W1 [64][192], W2T [64][192] (W2 transposed), b1 [64], b2 [192]; rows h >= H stay zero.
// Per step: x from a counter-based hash (the generator is stated below), s = max |x_u|,
// forward, residual, back-propagation (complex gradients as d/dRe + j d/dIm of the
// real loss; the Cartesian ReLU passes the real and the imaginary part of the hidden
// gradient where the real and the imaginary part of the pre-activation are positive),
// Adam on the real and imaginary parts with a cosine-decayed step size.  Every
// `eval_every` steps e^u is measured on a fixed test set of 64 samples; training of the
// network stops once it is below the tolerance or after `max_steps`.
#include <algorithm>
#include <array>
#include <chrono>
#include <map>
#include <vector>

#include "ie_internal.h"

namespace ie {
namespace {

constexpr int kTB = 32;             // minibatch
constexpr int kTP = kTB + 2;        // padded row length (float2)
constexpr int kTK = 16;             // rows of a chunk of a 192-row product's matrix
constexpr int kTC = 32;             // columns of a chunk of a 64-row product's matrix
constexpr int kTCP = kTC + 2;
constexpr int kTrainThreads = 256;
constexpr int kTestSamples = 64;
constexpr int kWElems = kCvHp * kNU;                    // W1 or W2T
constexpr int kStateElems = 2 * kWElems + kCvHp + kNU;  // W1, W2T, b1, b2
constexpr uint32_t kTestStream = 0xFFFFFFFFu;           // step index of the test set

struct SmemTrain {
    float2 X[kNU][kTP];
    float2 R[kNU][kTP];
    float2 Z[kCvHp][kTP];
    float2 Hh[kCvHp][kTP];
    union {
        float2 big[2][kTK][kNU];
        float2 hid[2][kCvHp][kTCP];
    } A;
    float inv_s[kTB];
    float red[kTrainThreads / 32];
    float err[kTB];
    float enorm[kTB];
};

// splitmix64 finaliser: the counter-based generator of the training inputs
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
// two uniforms in [-1, 1) from one draw
__device__ __forceinline__ float2 uniform2(uint64_t seed, uint32_t net, uint32_t step, uint32_t idx) {
    const uint64_t r = mix64(seed ^ mix64(((uint64_t)net << 32 | step) ^ mix64(idx)));
    const float a = (float)(r >> 40) * (1.0f / 16777216.0f);             // 24 bits
    const float b = (float)((r >> 16) & 0xFFFFFF) * (1.0f / 16777216.0f);
    return make_float2(2.f * a - 1.f, 2.f * b - 1.f);
}
// standard normal pair by Box-Muller from one draw
__device__ __forceinline__ float2 normal2(uint64_t seed, uint32_t net, uint32_t idx) {
    const uint64_t r = mix64(seed ^ mix64(((uint64_t)net << 32 | 0xABCDu) ^ mix64(idx)));
    const float u1 = ((float)(r >> 40) + 1.f) * (1.0f / 16777217.0f);
    const float u2 = (float)((r >> 16) & 0xFFFFFF) * (1.0f / 16777216.0f);
    const float rad = sqrtf(-2.f * logf(u1));
    float sn, cs;
    sincosf(6.2831853f * u2, &sn, &cs);
    return make_float2(rad * cs, rad * sn);
}

__device__ __forceinline__ void cfma(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}

struct TrainArgs {
    const float2 *C;        // [net][192 k][192 m] FP32 blocks G_c (transposed)
    float2 *state;          // [net][4][kStateElems]: weights, Adam m, Adam v ((re, im) second moments),
                            // gradient sum over the minibatches of a step
    float2 *Wout;           // [net][kCvBlockElems] trained networks in the inference layout
    float *eu;              // [net] final e^u
    int *steps_used;        // [net]
    int64_t nnet;
    int H, max_steps, eval_every, micro;
    float lr, tol;
    uint64_t seed;
};

// Inputs of a minibatch (or half of the test set) into S.X and their 1 / s.
__device__ void make_inputs(SmemTrain &S, const TrainArgs &a, uint32_t net, uint32_t step, int part) {
    const int t = threadIdx.x;
    for (int idx = t; idx < kNU * kTB; idx += kTrainThreads) {
        const int u = idx / kTB, j = idx % kTB;
        S.X[u][j] = uniform2(a.seed, net, step, (uint32_t)((part * kTB + j) * kNU + u));
    }
    __syncthreads();
    // s_j = max_u |x_u|: warp w reduces samples w, w + 8, w + 16, w + 24
    const int w = t >> 5, lane = t & 31;
    for (int j = w; j < kTB; j += kTrainThreads / 32) {
        float m = 0.f;
        for (int u = lane; u < kNU; u += 32) {
            const float2 x = S.X[u][j];
            m = fmaxf(m, x.x * x.x + x.y * x.y);
        }
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) S.inv_s[j] = m > 0.f ? rsqrtf(m) : 0.f;
    }
    __syncthreads();
    for (int idx = t; idx < kNU * kTB; idx += kTrainThreads) {
        const int u = idx / kTB, j = idx % kTB;
        const float q = S.inv_s[j];
        S.X[u][j] = make_float2(S.X[u][j].x * q, S.X[u][j].y * q);
    }
    __syncthreads();
}

__device__ __forceinline__ void copy16(void *smem, const void *gmem) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void copies_end() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// acc[i][c] += sum_k A[k][row i] B[k][column c], k < K <= 192, A [K][192] in global memory
// (whole chunks of 16 rows readable), B in shared memory.  Thread: rows 2 tm, + 1 (+ 64 i),
// columns 4 tn .. + 3, tm = t / 8, tn = t mod 8.  Ends with a barrier.
__device__ __forceinline__ void product192(SmemTrain &S, const float2 *A, int K, const float2 (*B)[kTP],
                                           float2 (&acc)[6][4]) {
    const int t = threadIdx.x, tm = t >> 3, tn = t & 7, chunks = (K + kTK - 1) / kTK;
    auto load = [&](int c) {
        const float4 *g = reinterpret_cast<const float4 *>(A + (size_t)c * kTK * kNU);
        float4 *d = reinterpret_cast<float4 *>(&S.A.big[c & 1][0][0]);
#pragma unroll
        for (int i = 0; i < kTK * kNU / 2 / kTrainThreads; ++i) copy16(d + t + i * kTrainThreads, g + t + i * kTrainThreads);
        copies_end();
    };
    load(0);
    for (int c = 0; c < chunks; ++c) {
        if (c + 1 < chunks) {
            load(c + 1);
            copies_wait<1>();
        } else {
            copies_wait<0>();
        }
        __syncthreads();
        const int kn = min(kTK, K - c * kTK);
#pragma unroll 2
        for (int k = 0; k < kn; ++k) {
            float2 a[6], b[4];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(&S.A.big[c & 1][k][2 * tm + 64 * i]);
                a[2 * i] = make_float2(v.x, v.y);
                a[2 * i + 1] = make_float2(v.z, v.w);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(&B[c * kTK + k][4 * tn + 2 * i]);
                b[2 * i] = make_float2(v.x, v.y);
                b[2 * i + 1] = make_float2(v.z, v.w);
            }
#pragma unroll
            for (int i = 0; i < 6; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) cfma(acc[i][q], a[i], b[q]);
        }
        __syncthreads();
    }
}
__device__ __forceinline__ int row192(int i) { return 2 * (threadIdx.x >> 3) + 64 * (i >> 1) + (i & 1); }
__device__ __forceinline__ int col192(int q) { return 4 * (threadIdx.x & 7) + q; }

// acc[r][c] = sum_k A[row r][k] B[k][column c] (CONJ: conj(A)), k < 192, A [64][192] in global
// memory, B in shared memory.  Thread: rows t / 16 + 16 r (below H), columns 2 (t mod 16), + 1.
// Ends with a barrier.
template <bool CONJ>
__device__ __forceinline__ void product64(SmemTrain &S, const float2 *A, int H, const float2 (*B)[kTP],
                                          float2 (&acc)[4][2]) {
    const int t = threadIdx.x, hg = t >> 4, jp = 2 * (t & 15);
    auto load = [&](int c) {
#pragma unroll
        for (int i = 0; i < kCvHp * kTC / 2 / kTrainThreads; ++i) {
            const int e = t + i * kTrainThreads, h = e / (kTC / 2), k = 2 * (e % (kTC / 2));
            copy16(&S.A.hid[c & 1][h][k], A + (size_t)h * kNU + c * kTC + k);
        }
        copies_end();
    };
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
    load(0);
    for (int c = 0; c < kNU / kTC; ++c) {
        if (c + 1 < kNU / kTC) {
            load(c + 1);
            copies_wait<1>();
        } else {
            copies_wait<0>();
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < kTC; k += 2) {
            const float4 x0 = *reinterpret_cast<const float4 *>(&B[c * kTC + k][jp]);
            const float4 x1 = *reinterpret_cast<const float4 *>(&B[c * kTC + k + 1][jp]);
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (hg + 16 * r < H) {
                    const float4 w = *reinterpret_cast<const float4 *>(&S.A.hid[c & 1][hg + 16 * r][k]);
                    const float2 b[2][2] = {{make_float2(x0.x, x0.y), make_float2(x0.z, x0.w)},
                                            {make_float2(x1.x, x1.y), make_float2(x1.z, x1.w)}};
                    const float2 a[2] = {make_float2(w.x, w.y), make_float2(w.z, w.w)};
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            if (CONJ) {
                                acc[r][q].x = fmaf(a[e].x, b[e][q].x, fmaf(a[e].y, b[e][q].y, acc[r][q].x));
                                acc[r][q].y = fmaf(a[e].x, b[e][q].y, fmaf(-a[e].y, b[e][q].x, acc[r][q].y));
                            } else {
                                cfma(acc[r][q], a[e], b[e][q]);
                            }
                        }
                }
        }
        __syncthreads();
    }
}

// R[m][j] = sum_k G[m][k] X[k][j] / g
__device__ void teacher(SmemTrain &S, const float2 *__restrict__ G, float ginv) {
    float2 acc[6][4];
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = make_float2(0.f, 0.f);
    product192(S, G, kNU, S.X, acc);
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) S.R[row192(i)][col192(c)] = make_float2(acc[i][c].x * ginv, acc[i][c].y * ginv);
}

// Z = W1 X + b1, Hh = relu(Z)
__device__ void forward_hidden(SmemTrain &S, const float2 *W1, const float2 *b1, int H) {
    float2 acc[4][2];
    product64<false>(S, W1, H, S.X, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int h = (threadIdx.x >> 4) + 16 * r;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int j = 2 * (threadIdx.x & 15) + q;
            float2 z = make_float2(0.f, 0.f);
            if (h < H) z = make_float2(acc[r][q].x + b1[h].x, acc[r][q].y + b1[h].y);
            S.Z[h][j] = z;
            S.Hh[h][j] = make_float2(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f));
        }
    }
}

// out[m][j] = W2 Hh + b2; mode 0: R = c (out - R); mode 1: per-sample |out - R|^2 and |R|^2
// into S.err / S.enorm (test set)
__device__ void forward_output(SmemTrain &S, const float2 *W2T, const float2 *b2, int H, float c, int mode) {
    float2 acc[6][4];
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = b2[row192(i)];
    product192(S, W2T, H, S.Hh, acc);
    if (mode == 0) {
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float2 &r = S.R[row192(i)][col192(q)];
                r = make_float2(c * (acc[i][q].x - r.x), c * (acc[i][q].y - r.y));
            }
    } else {
        float e[4] = {0.f, 0.f, 0.f, 0.f}, n[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 r = S.R[row192(i)][col192(q)];
                const float dx = acc[i][q].x - r.x, dy = acc[i][q].y - r.y;
                e[q] += dx * dx + dy * dy;
                n[q] += r.x * r.x + r.y * r.y;
            }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            atomicAdd(&S.err[col192(q)], e[q]);
            atomicAdd(&S.enorm[col192(q)], n[q]);
        }
    }
}

// g[r][i] = sum_j a_rj conj(b_ij) over the 32 samples for rows h = warp + 8 r < H of `rows` and
// entries u = lane + 32 i of `cols`; swap: the entries are the rows' conjugates' partner, i.e.
// sum_j cols[u][j] conj(rows[h][j]).
template <bool SWAP, class F>
__device__ __forceinline__ void gradient(const float2 (*rows)[kTP], const float2 (*cols)[kTP], int H, F use) {
    constexpr int kR = kCvHp / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // two halves of the rows: 4 x 6 sums in registers at a time
#pragma unroll 1
    for (int r0 = 0; r0 < kR; r0 += kR / 2) {
        if (warp + 8 * r0 >= H) break;
        float2 g[kR / 2][kNU / 32];
#pragma unroll
        for (int r = 0; r < kR / 2; ++r)
#pragma unroll
            for (int i = 0; i < kNU / 32; ++i) g[r][i] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int j = 0; j < kTB; j += 2) {
            float4 b[kNU / 32];
#pragma unroll
            for (int i = 0; i < kNU / 32; ++i) b[i] = *reinterpret_cast<const float4 *>(&cols[lane + 32 * i][j]);
#pragma unroll
            for (int r = 0; r < kR / 2; ++r)
                if (warp + 8 * (r0 + r) < H) {
                    const float4 h = *reinterpret_cast<const float4 *>(&rows[warp + 8 * (r0 + r)][j]);
#pragma unroll
                    for (int i = 0; i < kNU / 32; ++i) {
                        float2 &q = g[r][i];
                        if (SWAP) {         // cols conj(rows)
                            q.x = fmaf(b[i].x, h.x, fmaf(b[i].y, h.y, q.x));
                            q.y = fmaf(b[i].y, h.x, fmaf(-b[i].x, h.y, q.y));
                            q.x = fmaf(b[i].z, h.z, fmaf(b[i].w, h.w, q.x));
                            q.y = fmaf(b[i].w, h.z, fmaf(-b[i].z, h.w, q.y));
                        } else {            // rows conj(cols)
                            q.x = fmaf(h.x, b[i].x, fmaf(h.y, b[i].y, q.x));
                            q.y = fmaf(h.y, b[i].x, fmaf(-h.x, b[i].y, q.y));
                            q.x = fmaf(h.z, b[i].z, fmaf(h.w, b[i].w, q.x));
                            q.y = fmaf(h.w, b[i].z, fmaf(-h.z, b[i].w, q.y));
                        }
                    }
                }
        }
#pragma unroll
        for (int r = 0; r < kR / 2; ++r)
            if (warp + 8 * (r0 + r) < H) use((warp + 8 * (r0 + r)) * kNU + lane, g[r]);
    }
}

// Adam on one complex parameter (real and imaginary parts separately)
__device__ __forceinline__ void adam(float2 &p, float2 &m, float2 &v, float2 g, float lr_t, float c1, float c2) {
    constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    m = make_float2(b1 * m.x + (1.f - b1) * g.x, b1 * m.y + (1.f - b1) * g.y);
    v = make_float2(b2 * v.x + (1.f - b2) * g.x * g.x, b2 * v.y + (1.f - b2) * g.y * g.y);
    p.x -= lr_t * (m.x * c1) / (sqrtf(v.x * c2) + eps);
    p.y -= lr_t * (m.y * c1) / (sqrtf(v.y * c2) + eps);
}

// The gradient of one minibatch: summed into gs, or (last minibatch of the step) the
// sum taken and the Adam step made.
__device__ __forceinline__ void accumulate(float2 &p, float2 &m, float2 &v, float2 &gs, float2 g, bool first, bool last,
                                           float lr_t, float c1, float c2) {
    if (!first) g = make_float2(g.x + gs.x, g.y + gs.y);
    if (last)
        adam(p, m, v, g, lr_t, c1, c2);
    else
        gs = g;
}

// The same for the six entries at idx + 32 i of one row: all their reads are in flight before
// the first store.
__device__ __forceinline__ void accumulate_row(float2 *P, float2 *M, float2 *V, float2 *Gs, int idx,
                                               const float2 (&g)[kNU / 32], bool first, bool last, float lr_t, float c1,
                                               float c2) {
    constexpr int N = kNU / 32;
    float2 gs[N], p[N], m[N], v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (!first) gs[i] = Gs[idx + 32 * i];
        if (last) p[i] = P[idx + 32 * i], m[i] = M[idx + 32 * i], v[i] = V[idx + 32 * i];
    }
#pragma unroll
    for (int i = 0; i < N; ++i) accumulate(p[i], m[i], v[i], gs[i], g[i], first, last, lr_t, c1, c2);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (last)
            P[idx + 32 * i] = p[i], M[idx + 32 * i] = m[i], V[idx + 32 * i] = v[i];
        else
            Gs[idx + 32 * i] = gs[i];
    }
}

__global__ void __launch_bounds__(kTrainThreads, 1) cvfcnn_train_kernel(const TrainArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmemTrain &S = *reinterpret_cast<SmemTrain *>(smem_raw);
    const int t = threadIdx.x;
    const int H = a.H;
    for (int64_t net = blockIdx.x; net < a.nnet; net += gridDim.x) {
        const float2 *G = a.C + (size_t)net * kNU * kNU;
        float2 *P = a.state + (size_t)net * 4 * kStateElems;
        float2 *M = P + kStateElems, *V = M + kStateElems, *Gs = V + kStateElems;
        float2 *W1 = P, *W2T = P + kWElems, *b1 = P + 2 * kWElems, *b2 = b1 + kCvHp;
        // g = max |G_c|
        float gm = 0.f;
        for (int i = t; i < kNU * kNU; i += kTrainThreads) {
            const float2 v = G[i];
            gm = fmaxf(gm, v.x * v.x + v.y * v.y);
        }
        for (int o = 16; o; o >>= 1) gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
        if ((t & 31) == 0) S.red[t >> 5] = gm;
        __syncthreads();
        float g2 = 0.f;
        for (int w = 0; w < kTrainThreads / 32; ++w) g2 = fmaxf(g2, S.red[w]);
        const float gscale = g2 > 0.f ? sqrtf(g2) : 1.f, ginv = 1.f / gscale;
        // initial weights: W1 ~ CN(0, 1/192), W2 ~ CN(0, 1/H), biases 0; moments 0
        for (int i = t; i < kStateElems; i += kTrainThreads) {
            float2 w = make_float2(0.f, 0.f);
            if (i < kWElems) {
                if (i / kNU < H) {
                    const float2 z = normal2(a.seed, (uint32_t)net, (uint32_t)i);
                    const float sd = rsqrtf(2.f * kNU);
                    w = make_float2(z.x * sd, z.y * sd);
                }
            } else if (i < 2 * kWElems) {
                if ((i - kWElems) / kNU < H) {
                    const float2 z = normal2(a.seed, (uint32_t)net, (uint32_t)i);
                    const float sd = rsqrtf(2.f * H);
                    w = make_float2(z.x * sd, z.y * sd);
                }
            }
            P[i] = w;
            M[i] = make_float2(0.f, 0.f);
            V[i] = make_float2(0.f, 0.f);
        }
        __syncthreads();
        float eu = 1.f;
        int step = 0;
        const float cres = 2.f / (kTB * kNU);
        for (; step < a.max_steps; ++step) {
            if (a.eval_every > 0 && step % a.eval_every == 0 && step > 0) {
                // e^u on the test set (two halves of 32)
                float acc = 0.f;
                for (int part = 0; part < kTestSamples / kTB; ++part) {
                    make_inputs(S, a, (uint32_t)net, kTestStream, part);
                    teacher(S, G, ginv);
                    if (t < kTB) S.err[t] = S.enorm[t] = 0.f;
                    __syncthreads();
                    forward_hidden(S, W1, b1, H);
                    __syncthreads();
                    forward_output(S, W2T, b2, H, 0.f, 1);
                    __syncthreads();
                    if (t < 32) {
                        float v = S.enorm[t] > 0.f ? sqrtf(S.err[t] / S.enorm[t]) : 0.f;
                        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                        if (t == 0) S.red[0] = v;
                    }
                    __syncthreads();
                    acc += S.red[0];
                    __syncthreads();
                }
                eu = acc / kTestSamples;
                if (eu < a.tol) break;
            }
            const float lr_t = a.lr * (0.02f + 0.98f * 0.5f * (1.f + cospif((float)step / (float)a.max_steps)));
            const float c1 = 1.f / (1.f - powf(0.9f, (float)(step + 1)));
            const float c2 = 1.f / (1.f - powf(0.999f, (float)(step + 1)));
            // one Adam step on the gradient summed over `micro` minibatches of 32, all
            // taken with the weights of the start of the step
            for (int mbt = 0; mbt < a.micro; ++mbt) {
            const bool first = mbt == 0, last = mbt == a.micro - 1;
            make_inputs(S, a, (uint32_t)net, (uint32_t)(step * a.micro + mbt), 0);
            teacher(S, G, ginv);
            __syncthreads();
            forward_hidden(S, W1, b1, H);
            __syncthreads();
            forward_output(S, W2T, b2, H, cres, 0);
            __syncthreads();
            // hidden gradient with the old W2: dH = W2^H R, then dZ = dH through the ReLU (into Z)
            {
                float2 acc[4][2];
                product64<true>(S, W2T, H, S.R, acc);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int h = (t >> 4) + 16 * r, j = 2 * (t & 15) + q;
                        const float2 z = S.Z[h][j];
                        S.Z[h][j] = make_float2(z.x > 0.f ? acc[r][q].x : 0.f, z.y > 0.f ? acc[r][q].y : 0.f);
                    }
            }
            // W2 (transposed) and b2: dW2T[k][m] = sum_j R[m][j] conj(Hh[k][j])
            gradient<true>(S.Hh, S.R, H, [&](int idx, const float2 (&g)[kNU / 32]) {
                accumulate_row(P, M, V, Gs, kWElems + idx, g, first, last, lr_t, c1, c2);
            });
            for (int m = t; m < kNU; m += kTrainThreads) {
                float2 g = make_float2(0.f, 0.f);
                for (int j = 0; j < kTB; ++j) g = make_float2(g.x + S.R[m][j].x, g.y + S.R[m][j].y);
                const int o = 2 * kWElems + kCvHp + m;
                accumulate(b2[m], M[o], V[o], Gs[o], g, first, last, lr_t, c1, c2);
            }
            __syncthreads();
            // W1 and b1: dW1[h][u] = sum_j dZ[h][j] conj(X[u][j])
            gradient<false>(S.Z, S.X, H, [&](int idx, const float2 (&g)[kNU / 32]) {
                accumulate_row(P, M, V, Gs, idx, g, first, last, lr_t, c1, c2);
            });
            for (int h = t; h < H; h += kTrainThreads) {
                float2 g = make_float2(0.f, 0.f);
                for (int j = 0; j < kTB; ++j) g = make_float2(g.x + S.Z[h][j].x, g.y + S.Z[h][j].y);
                accumulate(b1[h], M[2 * kWElems + h], V[2 * kWElems + h], Gs[2 * kWElems + h], g, first, last, lr_t,
                           c1, c2);
            }
            __syncthreads();
            }
        }
        // e^u of the final weights (if the loop ran out before a check)
        if (step >= a.max_steps) {
            float acc = 0.f;
            for (int part = 0; part < kTestSamples / kTB; ++part) {
                make_inputs(S, a, (uint32_t)net, kTestStream, part);
                teacher(S, G, ginv);
                if (t < kTB) S.err[t] = S.enorm[t] = 0.f;
                __syncthreads();
                forward_hidden(S, W1, b1, H);
                __syncthreads();
                forward_output(S, W2T, b2, H, 0.f, 1);
                __syncthreads();
                if (t < 32) {
                    float v = S.enorm[t] > 0.f ? sqrtf(S.err[t] / S.enorm[t]) : 0.f;
                    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    if (t == 0) S.red[0] = v;
                }
                __syncthreads();
                acc += S.red[0];
                __syncthreads();
            }
            eu = acc / kTestSamples;
        }
        // the network in the inference layout: W1^T [192][64], b1, W2^T [64][192] and b2 times g
        float2 *O = a.Wout + (size_t)net * kCvBlockElems;
        for (int idx = t; idx < kWElems; idx += kTrainThreads) {
            const int h = idx / kNU, u = idx % kNU;
            O[kCvW1 + (size_t)u * kCvHp + h] = W1[idx];
            const float2 w2 = W2T[idx];
            O[kCvW2 + idx] = make_float2(w2.x * gscale, w2.y * gscale);
        }
        for (int h = t; h < kCvHp; h += kTrainThreads) O[kCvB1 + h] = b1[h];
        for (int m = t; m < kNU; m += kTrainThreads) O[kCvB2 + m] = make_float2(b2[m].x * gscale, b2[m].y * gscale);
        if (t == 0) {
            a.eu[net] = eu;
            a.steps_used[net] = step;
        }
        __syncthreads();
    }
}

}  // namespace

ie_status launch_cvfcnn_train(ie_plan p, const ie_cvfcnn_train_opts &o, ie_cvfcnn_train_info *info, cudaStream_t st) {
    auto t0 = std::chrono::steady_clock::now();
    // canonical displacements of the plan's far groups, and each group's block and frame
    std::vector<int32_t> canon, gcanon(p->n_far_disp), gsigma(p->n_far_disp);
    {
        std::map<std::array<int32_t, 3>, int32_t> index;
        for (int64_t d = 0; d < p->n_far_disp; ++d) {
            int32_t c[3];
            gsigma[d] = canon_of_disp(&p->h_disp[3 * d], c);
            auto ins = index.emplace(std::array<int32_t, 3>{c[0], c[1], c[2]}, (int32_t)index.size());
            if (ins.second) canon.insert(canon.end(), c, c + 3);
            gcanon[d] = ins.first->second;
        }
    }
    const int64_t ncanon = (int64_t)canon.size() / 3;
    if (info) *info = ie_cvfcnn_train_info{};
    if (ncanon == 0) return IE_OK;
    // with the symmetric store the stored blocks are these canonical ones, in this order
    if (p->sym && ncanon != p->n_blocks) return set_error("canonical blocks do not match the store"), IE_ERR_CUDA;
    int32_t *d_canon = nullptr, *d_gc = nullptr, *d_gs = nullptr, *d_steps = nullptr;
    float2 *C = nullptr, *state = nullptr, *Wc = nullptr;
    float *d_eu = nullptr;
    uint16_t *d_map = nullptr;
    std::vector<uint16_t> map;
    symmetry_map_host(map);
    ie_status s = IE_OK;
    auto ck = [&](cudaError_t e, const char *what) {
        if (e != cudaSuccess && s == IE_OK) {
            cudaGetLastError();
            set_error("CVFCNN training %s: %s", what, cudaGetErrorString(e));
            s = e == cudaErrorMemoryAllocation ? IE_ERR_OOM : IE_ERR_CUDA;
        }
    };
    ck(cudaMallocAsync(&d_canon, canon.size() * sizeof(int32_t), st), "scratch");
    ck(cudaMallocAsync(&C, (size_t)ncanon * kNU * kNU * sizeof(float2), st), "scratch");
    ck(cudaMallocAsync(&state, (size_t)ncanon * 4 * kStateElems * sizeof(float2), st), "scratch");
    ck(cudaMallocAsync(&d_eu, (size_t)ncanon * sizeof(float), st), "scratch");
    ck(cudaMallocAsync(&d_steps, (size_t)ncanon * sizeof(int), st), "scratch");
    if (!p->sym) {
        ck(cudaMallocAsync(&Wc, (size_t)ncanon * kCvBlockElems * sizeof(float2), st), "scratch");
        ck(cudaMallocAsync(&d_gc, gcanon.size() * sizeof(int32_t), st), "scratch");
        ck(cudaMallocAsync(&d_gs, gsigma.size() * sizeof(int32_t), st), "scratch");
        ck(cudaMallocAsync(&d_map, map.size() * sizeof(uint16_t), st), "scratch");
    }
    if (s == IE_OK) {
        ck(cudaMemcpyAsync(d_canon, canon.data(), canon.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st), "copy");
        if (!p->sym) {
            ck(cudaMemcpyAsync(d_gc, gcanon.data(), gcanon.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st), "copy");
            ck(cudaMemcpyAsync(d_gs, gsigma.data(), gsigma.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st), "copy");
            ck(cudaMemcpyAsync(d_map, map.data(), map.size() * sizeof(uint16_t), cudaMemcpyHostToDevice, st), "copy");
        }
    }
    if (s == IE_OK) s = launch_coupling_simt(p, d_canon, ncanon, C, false, st);   // G_c, FP64 -> FP32, [k][m]
    if (s == IE_OK) {
        TrainArgs a;
        a.C = C;
        a.state = state;
        a.Wout = p->sym ? p->d_cvW : Wc;
        a.eu = d_eu;
        a.steps_used = d_steps;
        a.nnet = ncanon;
        a.H = p->cv_hidden;
        a.max_steps = o.max_steps;
        a.eval_every = o.eval_every;
        a.micro = o.minibatches;
        a.lr = (float)o.lr;
        a.tol = (float)o.tol;
        a.seed = o.seed;
        int dev = 0, sms = 0;
        ck(cudaGetDevice(&dev), "device");
        ck(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "device");
        if (s == IE_OK) {
            const int grid = (int)std::min<int64_t>(ncanon, sms);
            cvfcnn_train_kernel<<<grid, kTrainThreads, sizeof(SmemTrain), st>>>(a);
            count_launches(1);
            ck(cudaGetLastError(), "launch");
        }
    }
    if (s == IE_OK && !p->sym) {
        launch_cvfcnn_expand(Wc, d_gc, d_gs, d_map, p->n_blocks, p->d_cvW, st);
        ck(cudaGetLastError(), "expansion");
    }
    if (s == IE_OK) s = build_cvfcnn_images(p, st);
    std::vector<float> eu(ncanon);
    std::vector<int> steps(ncanon);
    if (s == IE_OK) {
        ck(cudaMemcpyAsync(eu.data(), d_eu, ncanon * sizeof(float), cudaMemcpyDeviceToHost, st), "copy");
        ck(cudaMemcpyAsync(steps.data(), d_steps, ncanon * sizeof(int), cudaMemcpyDeviceToHost, st), "copy");
        ck(cudaStreamSynchronize(st), "sync");
    }
    for (void *ptr : {(void *)d_canon, (void *)C, (void *)state, (void *)d_eu, (void *)d_steps, (void *)Wc, (void *)d_gc,
                      (void *)d_gs, (void *)d_map})
        if (ptr) cudaFreeAsync(ptr, st);
    if (s != IE_OK) return s;
    if (info) {
        info->networks = ncanon;
        double mx = 0, mean = 0;
        int below = 0, smax = 0;
        for (int64_t i = 0; i < ncanon; ++i) {
            mx = std::max(mx, (double)eu[i]);
            mean += eu[i];
            below += eu[i] < o.tol ? 1 : 0;
            smax = std::max(smax, steps[i]);
        }
        info->eu_max = mx;
        info->eu_mean = mean / ncanon;
        info->converged = below;
        info->steps_max = smax;
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    p->cv_trained = 1;
    return IE_OK;
}

ie_status prepare_cvfcnn_train() {
    IE_CK(cudaFuncSetAttribute(cvfcnn_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(SmemTrain)));
    return IE_OK;
}

}  // namespace ie

using namespace ie;

extern "C" void ie_cvfcnn_train_opts_default(ie_cvfcnn_train_opts *o) {
    if (!o) return;
    o->max_steps = 8000;
    o->minibatches = 4;
    o->eval_every = 250;
    o->lr = 4e-3;
    o->tol = 1e-3;
    o->seed = 20250108;
}

extern "C" ie_status ie_cvfcnn_train(ie_plan p, const ie_cvfcnn_train_opts *opts, ie_cvfcnn_train_info *info,
                                     void *stream) {
    ie::NvtxRange nvtx_range("ie_cvfcnn_train");
    if (!p) return set_error("null plan"), IE_ERR_INVALID;
    if (!p->d_cvW) return set_error("the plan holds no CVFCNN surrogates"), IE_ERR_UNSUPPORTED;
    ie_cvfcnn_train_opts o;
    ie_cvfcnn_train_opts_default(&o);
    if (opts) o = *opts;
    if (o.max_steps < 0 || o.max_steps > 1000000 || o.minibatches < 1 || o.minibatches > 64 || o.eval_every < 0 ||
        !(o.lr > 0) || !(o.tol > 0))
        return set_error("bad training options"), IE_ERR_INVALID;
    IE_TRY(prepare_cvfcnn_train());
    return launch_cvfcnn_train(p, o, info, (cudaStream_t)stream);
}

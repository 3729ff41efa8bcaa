// K6 / K8: restarted GMRES without preconditioning (§5, the paper's iterative
// solver) with device-resident state, and outer iterative refinement.
//
// Systems: every (right-hand side, scatterer) pair is an independent GMRES(m) run
// (x0 = 0) over its scatterer's slice of the packed vector [rhs][n]; a plan without
// scatterer groups has one system per right-hand side.  Arnoldi uses classical
// Gram-Schmidt applied twice (dot products accumulated in FP64), Givens rotations and
// the small least-squares solve run in FP64; Krylov vectors are FP32.  Vector kernels
// walk chunks of 512 unknowns that never straddle two scatterers.
//
// An iteration is the product and four kernels: each Gram-Schmidt pass's update and the next
// sums share a pass over W, and the last block of a system to arrive adds the chunks' sums
// (and rotates the new Hessenberg column), the last of all advances the loop.  Bound by the
// kernels' latencies: 10 launches took 65 us beside the product on the 16^3 shell, these 4 take
// 35 us (solve of nine products 1,843 -> 1,584 us).
// One restart cycle is one CUDA graph: a WHILE node runs one Arnoldi iteration per
// body launch (the iteration index lives in device memory and the Givens kernel sets
// the condition from the per-system flags), followed by the solution update and the
// restart residual.  The host synchronises once per cycle.
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "ie_internal.h"

struct ie_solver_s {
    ie_plan plan = nullptr;
    int R = 1, G = 1, S = 1, m = 50, max_iters = 1000, prec = IE_PREC_FP32;
    double tol = 1e-6;
    int64_t n = 0;
    int C = 1, nblk = 1;                 // chunks per column, max chunks of one scatterer
    int32_t *chunk_group = nullptr;      // [C]
    int64_t *chunk_start = nullptr;      // [C] first unknown of the chunk
    int32_t *chunk_local = nullptr;      // [C] chunk index inside its scatterer
    int64_t *goff = nullptr;             // [G + 1] unknown offsets of the scatterers
    int32_t *nchunk = nullptr;           // [G]
    float2 *V = nullptr;                 // [(m+1)][R][n]
    float2 *W = nullptr;                 // [R][n]
    float2 *Vcur = nullptr;              // [R][n] current Krylov vector (input of the product)
    double2 *H = nullptr;                // [S][m][m+1]
    double *cs = nullptr;                // [S][m]
    double2 *sn = nullptr;               // [S][m]
    double2 *g = nullptr;                // [S][m+1]
    double2 *hbuf = nullptr;             // [S][m+1]
    double2 *partial = nullptr;          // [S][m+1][nblk]
    double *bnorm = nullptr;             // [S]
    double *relres = nullptr;            // [S]
    int *st = nullptr;                   // [5 + 4S], layout below, relres behind it: one copy to the host
    int *cnt = nullptr;                  // [S + 1] block arrivals
    // outer refinement (first use): FP64 iterate, right-hand side, correction, product, sums
    double2 *x64 = nullptr, *rpart = nullptr, *h_part = nullptr;
    float2 *rv = nullptr, *rd = nullptr, *rw = nullptr;
    cudaGraphConditionalHandle hcond = 0;
    bool use_while = false;
    int64_t body_kernels = 0, end_kernels = 0, body_runs_seen = 0;
    const float2 *v = nullptr;
    float2 *x = nullptr;
    const float2 *cap_v = nullptr;       // pointers baked into the captured cycle
    float2 *cap_x = nullptr;
    cudaStream_t cap = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaEvent_t ev = nullptr;
    int matvecs_per_cycle = 0;
    int cycles_run = 0;
    int *h_st = nullptr;                 // pinned host mirror of st and relres, copied at the end of
    double *h_rel = nullptr;             // every start and advance (read by ie_solver_poll / _state)
    std::vector<void *> allocs;
    size_t bytes = 0;
};

namespace ie {
namespace {

constexpr int kDotThreads = 256;
// unknowns per thread in the vector kernels: small chunks spread the dot products' FP64 work
// (its rate bounds an SM) over more SMs; 1 / 2 / 4: 609 / 620 / 679 us (176 boxes, 3 columns), 1.48 /
// 1.45 / 1.52 ms (16^3 shell), 4.81 / 4.70 / 4.72 ms (32^3 shell) per solve
constexpr int kEPT = 2;
constexpr int kChunk = kDotThreads * kEPT;     // unknowns per chunk (one block)
constexpr int kMaxSystems = 1024;

// st layout: [0] any system active in this cycle, [1] any system not finished, then
// done[S], active[S], jend[S], iters[S], the cycle's Arnoldi index, WHILE-body runs, the
// plan's device error word at the start of the cycle.
inline __host__ __device__ int st_ints(int S) { return 5 + 4 * S; }
__device__ inline int *st_done(int *st, int S) { return st + 2; }
__device__ inline int *st_active(int *st, int S) { return st + 2 + S; }
__device__ inline int *st_jend(int *st, int S) { return st + 2 + 2 * S; }
__device__ inline int *st_iters(int *st, int S) { return st + 2 + 3 * S; }
__device__ inline int *st_jdev(int *st, int S) { return st + 2 + 4 * S; }
__device__ inline int *st_body(int *st, int S) { return st + 3 + 4 * S; }
__device__ inline int *st_err(int *st, int S) { return st + 4 + 4 * S; }

// j >= 0: index given by the launch; kDevJ: read the cycle's index from device memory.
constexpr int kDevJ = -2;
__device__ inline int resolve_j(int j, int *st, int S) { return j >= 0 ? j : *st_jdev(st, S); }

// Segmented layout of the packed vector.
struct Seg {
    const int32_t *chunk_group;
    const int64_t *chunk_start;
    const int32_t *chunk_local;
    const int64_t *goff;
    const int32_t *nchunk;
    int G;
    int64_t n;
};

// The system of chunk c in column r, the chunk's unknown range [e0, e1) and its
// index inside the scatterer.
__device__ inline int chunk_system(const Seg &sg, int c, int r, int64_t &e0, int64_t &e1, int &local) {
    const int g = sg.chunk_group[c];
    e0 = sg.chunk_start[c];
    e1 = min(e0 + (int64_t)kChunk, sg.goff[g + 1]);
    local = sg.chunk_local[c];
    return r * sg.G + g;
}

__device__ inline double2 block_sum2(double2 v) {
    __shared__ double2 red[kDotThreads / 32];
    for (int o = 16; o; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    int w = threadIdx.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double2 s = make_double2(0, 0);
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s.x += red[i].x, s.y += red[i].y;
    return s;   // valid in thread 0
}

__device__ inline double2 cmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ inline double2 conj2(double2 a) { return make_double2(a.x, -a.y); }
__device__ inline double cabs2(double2 a) { return sqrt(a.x * a.x + a.y * a.y); }

// The state one Arnoldi iteration works on.
struct Arnoldi {
    float2 *V, *W, *Vcur;
    Seg sg;
    int R, S, m, nblk;
    double2 *partial, *hbuf, *H, *sn, *g;
    double *cs, *relres;
    const double *bnorm;
    int *st;
    int *cnt;                   // [S + 1] arrivals of a system's chunks, of all chunks
    const int *err;             // the plan's device error word
    double tol;
    int max_iters;
};

// Counts the block in at cnt (all its global writes done) and tells whether it is the last of
// `total`; the last one then sees the others' writes.  The counter is left at zero.
__device__ inline bool last_block(int *cnt, int total) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(cnt, 1) == total - 1;
        if (s_last) *cnt = 0;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// pr[i][local] = the chunk's sum of conj(V_i) . w, i <= j.  Four vectors at a time: their
// reads are in flight together, and the tree halves the sums a lane carries (9 exchanges for
// eight sums instead of 40).
__device__ inline void chunk_dots(const float2 *__restrict__ Vr, int64_t vstride, const float2 (&w)[kEPT], int64_t e0,
                                  int64_t e1, int j, double2 *__restrict__ pr, int nblk, int local) {
    __shared__ double red[2][kDotThreads / 32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i0 = 0, buf = 0; i0 <= j; i0 += 4, buf ^= 1) {
        float2 a[4][kEPT];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int t = 0; t < kEPT; ++t) {
                const int64_t e = e0 + threadIdx.x + t * kDotThreads;
                a[q][t] = i0 + q <= j && e < e1 ? Vr[(i0 + q) * vstride + e] : make_float2(0.f, 0.f);
            }
        double v[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double sr = 0, si = 0;
            if (i0 + q <= j)
#pragma unroll
                for (int t = 0; t < kEPT; ++t) {
                    sr = fma((double)a[q][t].x, (double)w[t].x, fma((double)a[q][t].y, (double)w[t].y, sr));
                    si = fma((double)a[q][t].x, (double)w[t].y, fma(-(double)a[q][t].y, (double)w[t].x, si));
                }
            v[2 * q] = sr;
            v[2 * q + 1] = si;
        }
        int idx = 0;
#pragma unroll
        for (int o = 16, n = 4; o > 2; o >>= 1, n >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < n) {
                    const double send = up ? v[k] : v[k + n], keep = up ? v[k + n] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            idx += up ? n : 0;
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if ((lane & 3) == 0) red[buf][warp][idx] = v[0];
        __syncthreads();                        // two buffers: one barrier per four vectors
        if (threadIdx.x < 8 && i0 + (int)threadIdx.x / 2 <= j) {
            double sum = 0;
#pragma unroll
            for (int k = 0; k < kDotThreads / 32; ++k) sum += red[buf][k][threadIdx.x];
            reinterpret_cast<double *>(pr + (int64_t)(i0 + threadIdx.x / 2) * nblk + local)[threadIdx.x & 1] = sum;
        }
    }
}

// hbuf[i] = the sum of the system's chunks (warp per i); column j of H gets it (first
// Gram-Schmidt pass) or has it added (second pass).  By the system's last block.
__device__ inline void finish_dots(const Arnoldi &q, int s, int nb, int j, bool add) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i <= j; i += kDotThreads / 32) {
        const double2 *p = q.partial + ((int64_t)s * (q.m + 1) + i) * q.nblk;
        double sx = 0, sy = 0;
        for (int b = lane; b < nb; b += 32) {
            const double2 t = __ldcg(p + b);
            sx += t.x, sy += t.y;
        }
        for (int o = 16; o; o >>= 1) {
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if (lane == 0) {
            q.hbuf[(int64_t)s * (q.m + 1) + i] = make_double2(sx, sy);
            double2 &h = q.H[((int64_t)s * q.m + j) * (q.m + 1) + i];
            if (add) {
                h.x += sx;
                h.y += sy;
            } else {
                h = make_double2(sx, sy);
            }
        }
    }
}

// w -= sum_{i<=j} V_i hbuf[s][i] for the thread's unknowns of the chunk, stored in W.
__device__ inline void chunk_update(const Arnoldi &q, int s, int r, int64_t e0, int64_t e1, int j, float2 (&w)[kEPT]) {
    __shared__ float2 h[65];
    for (int i = threadIdx.x; i <= j; i += kDotThreads) {
        const double2 v = q.hbuf[(int64_t)s * (q.m + 1) + i];
        h[i] = make_float2((float)v.x, (float)v.y);
    }
    __syncthreads();
    const int64_t n = q.sg.n;
    float2 *wr = q.W + (int64_t)r * n;
#pragma unroll
    for (int t = 0; t < kEPT; ++t) {
        const int64_t e = e0 + threadIdx.x + t * kDotThreads;
        w[t] = e < e1 ? wr[e] : make_float2(0.f, 0.f);
    }
    const float2 *vr = q.V + (int64_t)r * n + e0 + threadIdx.x;
    for (int i = 0; i <= j; ++i) {
        const float2 hi = h[i];
        const float2 *vi = vr + (int64_t)i * q.R * n;
#pragma unroll
        for (int t = 0; t < kEPT; ++t)
            if (e0 + threadIdx.x + t * kDotThreads < e1) {
                const float2 a = vi[t * kDotThreads];
                w[t].x -= a.x * hi.x - a.y * hi.y;
                w[t].y -= a.x * hi.y + a.y * hi.x;
            }
    }
#pragma unroll
    for (int t = 0; t < kEPT; ++t) {
        const int64_t e = e0 + threadIdx.x + t * kDotThreads;
        if (e < e1) wr[e] = w[t];
    }
}

// First Gram-Schmidt pass: h_i = conj(V_i) . W.
__global__ void __launch_bounds__(kDotThreads) dots_kernel(const Arnoldi q, int jarg) {
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(q.sg, blockIdx.x, r, e0, e1, local);
    if (!st_active(q.st, q.S)[s]) return;
    const int j = resolve_j(jarg, q.st, q.S);
    float2 w[kEPT];
#pragma unroll
    for (int t = 0; t < kEPT; ++t) {
        const int64_t e = e0 + threadIdx.x + t * kDotThreads;
        w[t] = e < e1 ? q.W[(int64_t)r * q.sg.n + e] : make_float2(0.f, 0.f);
    }
    chunk_dots(q.V + (int64_t)r * q.sg.n, (int64_t)q.R * q.sg.n, w, e0, e1, j, q.partial + (int64_t)s * (q.m + 1) * q.nblk,
               q.nblk, local);
    const int nb = q.sg.nchunk[s % q.sg.G];
    if (last_block(q.cnt + s, nb)) finish_dots(q, s, nb, j, false);
}

// W -= sum h_i V_i, then the second pass's sums of the updated W.
__global__ void __launch_bounds__(kDotThreads) update_dots_kernel(const Arnoldi q, int jarg) {
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(q.sg, blockIdx.x, r, e0, e1, local);
    if (!st_active(q.st, q.S)[s]) return;
    const int j = resolve_j(jarg, q.st, q.S);
    float2 w[kEPT];
    chunk_update(q, s, r, e0, e1, j, w);
    chunk_dots(q.V + (int64_t)r * q.sg.n, (int64_t)q.R * q.sg.n, w, e0, e1, j, q.partial + (int64_t)s * (q.m + 1) * q.nblk,
               q.nblk, local);
    const int nb = q.sg.nchunk[s % q.sg.G];
    if (last_block(q.cnt + s, nb)) finish_dots(q, s, nb, j, true);
}

// Givens update of column j of one system, its residual estimate and termination; hn = ||W||.
// The column and the rotations are in shared memory (h, c, sv).  One thread.
__device__ inline void givens_column(const Arnoldi &q, int s, int j, double2 *h, double *c, double2 *sv) {
    double2 *gr = q.g + (int64_t)s * (q.m + 1);
    for (int i = 0; i < j; ++i) {
        double2 a = h[i], b = h[i + 1];
        double2 sb = cmul(sv[i], b);
        double2 u = cmul(conj2(sv[i]), a);
        h[i] = make_double2(c[i] * a.x + sb.x, c[i] * a.y + sb.y);
        h[i + 1] = make_double2(-u.x + c[i] * b.x, -u.y + c[i] * b.y);
    }
    double2 a = h[j], b = h[j + 1];
    double na = cabs2(a), nb = cabs2(b);
    double den = sqrt(na * na + nb * nb);
    double cj;
    double2 sj;
    if (den == 0) {
        cj = 1, sj = make_double2(0, 0);
    } else if (na == 0) {
        cj = 0, sj = make_double2(b.x / nb, -b.y / nb);
    } else {
        cj = na / den;
        double2 ph = make_double2(a.x / na, a.y / na);
        sj = cmul(ph, make_double2(b.x / den, -b.y / den));
    }
    q.cs[(int64_t)s * q.m + j] = cj;
    q.sn[(int64_t)s * q.m + j] = sj;
    double2 sb = cmul(sj, b);
    h[j] = make_double2(cj * a.x + sb.x, cj * a.y + sb.y);
    h[j + 1] = make_double2(0, 0);
    double2 gj = gr[j];
    double2 gn = cmul(conj2(sj), gj);
    gr[j + 1] = make_double2(-gn.x, -gn.y);
    gr[j] = make_double2(cj * gj.x, cj * gj.y);
    int it = ++st_iters(q.st, q.S)[s];
    st_jend(q.st, q.S)[s] = j + 1;
    double res = cabs2(gr[j + 1]) / q.bnorm[s];
    q.relres[s] = res;
    bool breakdown = nb == 0;
    if (res <= q.tol || it >= q.max_iters || breakdown || j + 1 == q.m) st_active(q.st, q.S)[s] = 0;
}

// The second pass's update, ||W|| and, by a system's last block, the Givens rotation of its
// column; the last block of all advances the iteration index and, in the WHILE body, sets the
// loop condition.
__global__ void __launch_bounds__(kDotThreads) update_norm_kernel(const Arnoldi q, int jarg,
                                                                  cudaGraphConditionalHandle cond) {
    __shared__ double2 s_h[66], s_sn[64];
    __shared__ double s_cs[64], s_norm;
    __shared__ int any;
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(q.sg, blockIdx.x, r, e0, e1, local);
    const int j = resolve_j(jarg, q.st, q.S);
    if (st_active(q.st, q.S)[s]) {
        float2 w[kEPT];
        chunk_update(q, s, r, e0, e1, j, w);
        double x = 0;
#pragma unroll
        for (int t = 0; t < kEPT; ++t) x += (double)w[t].x * w[t].x + (double)w[t].y * w[t].y;
        double2 *pr = q.partial + (int64_t)s * (q.m + 1) * q.nblk;
        const double2 tot = block_sum2(make_double2(x, 0));
        if (threadIdx.x == 0) pr[local] = tot;
        const int nb = q.sg.nchunk[s % q.sg.G];
        if (last_block(q.cnt + s, nb)) {
            double2 *H = q.H + ((int64_t)s * q.m + j) * (q.m + 1);
            if (threadIdx.x < 32) {
                double t = 0;
                for (int b = threadIdx.x; b < nb; b += 32) t += __ldcg(&pr[b].x);
                for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (threadIdx.x == 0) s_norm = sqrt(t);
            }
            for (int i = threadIdx.x; i <= j; i += kDotThreads) s_h[i] = H[i];
            for (int i = threadIdx.x; i < j; i += kDotThreads) {
                s_cs[i] = q.cs[(int64_t)s * q.m + i];
                s_sn[i] = q.sn[(int64_t)s * q.m + i];
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                s_h[j + 1] = make_double2(s_norm, 0);
                q.hbuf[(int64_t)s * (q.m + 1)] = make_double2(s_norm, 0);    // read by the scaling kernel
                givens_column(q, s, j, s_h, s_cs, s_sn);
            }
            __syncthreads();
            for (int i = threadIdx.x; i <= j + 1; i += kDotThreads) H[i] = s_h[i];
        }
    }
    if (!last_block(q.cnt + q.S, gridDim.x * gridDim.y)) return;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < q.S; k += kDotThreads)
        if (__ldcg(st_active(q.st, q.S) + k)) atomicOr(&any, 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        q.st[0] = any;
        if (jarg == kDevJ) {
            *st_jdev(q.st, q.S) = j + 1;
            *st_body(q.st, q.S) += 1;
            cudaGraphSetConditional(cond, any ? 1u : 0u);   // WHILE node: run the next iteration?
        }
    }
}

// V_{j+1} = W / hn over the chunk, also written to Vcur (the next product's input); systems
// that have just finished need neither.  The index has advanced: column j of V is the next one.
__global__ void __launch_bounds__(kDotThreads) scale_kernel(const Arnoldi q, int jnext) {
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(q.sg, blockIdx.x, r, e0, e1, local);
    if (!st_active(q.st, q.S)[s]) return;
    const int j = resolve_j(jnext, q.st, q.S);
    const double hn = q.hbuf[(int64_t)s * (q.m + 1)].x;
    const float f = hn > 0 ? (float)(1.0 / hn) : 0.f;
    const int64_t n = q.sg.n;
    const float2 *wr = q.W + (int64_t)r * n;
    float2 *vr = q.V + ((int64_t)j * q.R + r) * n;
    float2 *cr = q.Vcur + (int64_t)r * n;
#pragma unroll
    for (int t = 0; t < kEPT; ++t) {
        const int64_t e = e0 + threadIdx.x + t * kDotThreads;
        if (e >= e1) continue;
        const float2 w = wr[e];
        const float2 o = make_float2(w.x * f, w.y * f);
        vr[e] = o;
        cr[e] = o;
    }
}

// Back substitution H[0:jend,0:jend] y = g[0:jend] per system; y stored in hbuf[s].
__global__ void lsq_kernel(const double2 *__restrict__ H, const double2 *__restrict__ g, double2 *__restrict__ y,
                           int m, int S, int *st) {
    for (int s = threadIdx.x + blockIdx.x * blockDim.x; s < S; s += blockDim.x * gridDim.x) {
        const int je = st_jend(st, S)[s];
        double2 *ys = y + (int64_t)s * (m + 1);
        for (int i = je - 1; i >= 0; --i) {
            double2 q = g[(int64_t)s * (m + 1) + i];
            for (int k = i + 1; k < je; ++k) {
                double2 t = cmul(H[((int64_t)s * m + k) * (m + 1) + i], ys[k]);
                q.x -= t.x, q.y -= t.y;
            }
            double2 d = H[((int64_t)s * m + i) * (m + 1) + i];
            double dd = d.x * d.x + d.y * d.y;
            ys[i] = dd > 0 ? make_double2((q.x * d.x + q.y * d.y) / dd, (q.y * d.x - q.x * d.y) / dd)
                           : make_double2(0, 0);
        }
    }
}

// x += sum_{i<jend} V_i y[s][i] over the chunk
__global__ void xupdate_kernel(const float2 *__restrict__ V, float2 *__restrict__ x, Seg sg, int R, int S, int m,
                               const double2 *__restrict__ y, int *st) {
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(sg, blockIdx.x, r, e0, e1, local);
    const int je = st_jend(st, S)[s];
    if (je == 0) return;
    __shared__ float2 ys[65];
    for (int i = threadIdx.x; i < je; i += blockDim.x) {
        double2 v = y[(int64_t)s * (m + 1) + i];
        ys[i] = make_float2((float)v.x, (float)v.y);
    }
    __syncthreads();
    const int64_t n = sg.n;
    float2 *xr = x + (int64_t)r * n;
    for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        float2 acc = xr[e];
        for (int i = 0; i < je; ++i) {
            float2 a = V[((int64_t)i * R + r) * n + e];
            acc.x += a.x * ys[i].x - a.y * ys[i].y;
            acc.y += a.x * ys[i].y + a.y * ys[i].x;
        }
        xr[e] = acc;
    }
}

// Begin a cycle: V_0 = v - W over the chunk (W = Z x; start = 1: V_0 = v, x = 0) for systems
// not done, and by a system's last block beta = ||V_0||, the termination tests and g reset.
// start = 1 also sets bnorm = beta (x0 = 0).  The last block of all sets the cycle's flags.
__global__ void __launch_bounds__(kDotThreads) begin_cycle_kernel(const Arnoldi q, const float2 *__restrict__ v,
                                                                  float2 *__restrict__ x, int start,
                                                                  double *__restrict__ bnorm) {
    __shared__ int any;
    __shared__ double s_beta;
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(q.sg, blockIdx.x, r, e0, e1, local);
    if (start || !st_done(q.st, q.S)[s]) {
        const int64_t n = q.sg.n;
        double t2 = 0;
#pragma unroll
        for (int t = 0; t < kEPT; ++t) {
            const int64_t e = e0 + threadIdx.x + t * kDotThreads, i = (int64_t)r * n + e;
            if (e >= e1) continue;
            float2 a = v[i];
            if (start) {
                x[i] = make_float2(0.f, 0.f);
            } else {
                const float2 b = q.W[i];
                a.x -= b.x;
                a.y -= b.y;
            }
            q.V[i] = a;
            t2 += (double)a.x * a.x + (double)a.y * a.y;
        }
        double2 *pr = q.partial + (int64_t)s * (q.m + 1) * q.nblk;
        const double2 tot = block_sum2(make_double2(t2, 0));
        if (threadIdx.x == 0) pr[local] = tot;
        const int nb = q.sg.nchunk[s % q.sg.G];
        if (last_block(q.cnt + s, nb)) {
            if (threadIdx.x < 32) {
                double t = 0;
                for (int b = threadIdx.x; b < nb; b += 32) t += __ldcg(&pr[b].x);
                for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (threadIdx.x == 0) s_beta = sqrt(t);
            }
            __syncthreads();
            const double beta = s_beta;
            double2 *gr = q.g + (int64_t)s * (q.m + 1);
            for (int i = threadIdx.x; i <= q.m; i += kDotThreads) gr[i] = make_double2(i ? 0.0 : beta, 0);
            if (threadIdx.x == 0) {
                if (start) bnorm[s] = beta;
                const double bn = start ? beta : bnorm[s];
                const double rel = bn > 0 ? beta / bn : 0.0;
                q.relres[s] = rel;
                st_jend(q.st, q.S)[s] = 0;
                if (start) st_iters(q.st, q.S)[s] = 0;
                const bool fin = bn == 0 || rel <= q.tol || st_iters(q.st, q.S)[s] >= q.max_iters;
                st_done(q.st, q.S)[s] = fin;
                st_active(q.st, q.S)[s] = !fin;
                q.hbuf[(int64_t)s * (q.m + 1)] = make_double2(beta, 0);
            }
        }
    } else if (local == 0 && threadIdx.x == 0) {    // done before: nothing to update
        st_jend(q.st, q.S)[s] = 0;
        st_active(q.st, q.S)[s] = 0;
    }
    if (!last_block(q.cnt + q.S, gridDim.x * gridDim.y)) return;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < q.S; k += kDotThreads) {
        if (q.sg.nchunk[k % q.sg.G] == 0) {     // a scatterer without unknowns has no block
            st_done(q.st, q.S)[k] = 1;
            bnorm[k] = q.relres[k] = 0;
        }
        if (__ldcg(st_active(q.st, q.S) + k)) atomicOr(&any, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        q.st[0] = any;
        q.st[1] = any;   // a system not done is active at the start of a cycle
        *st_jdev(q.st, q.S) = 0;
        *st_err(q.st, q.S) = *q.err;
    }
}

// V_0 /= beta (hbuf[s][0]) over the chunk for active systems, also into Vcur.
__global__ void scale_v0_kernel(float2 *__restrict__ V0, float2 *__restrict__ Vcur, Seg sg, int S, int m,
                                const double2 *__restrict__ hbuf, int *st) {
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(sg, blockIdx.x, r, e0, e1, local);
    if (!st_active(st, S)[s]) return;
    const float q = (float)(1.0 / hbuf[(int64_t)s * (m + 1)].x);
    const int64_t n = sg.n;
    float2 *vr = V0 + (int64_t)r * n;
    float2 *cr = Vcur + (int64_t)r * n;
    for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        float2 a = vr[e];
        float2 o = make_float2(a.x * q, a.y * q);
        vr[e] = o;
        cr[e] = o;
    }
}

// ---- refinement helpers (FP64 outer loop) ----
// r = v - W in FP64 over the chunk; partial[s][local] = (||r||^2, ||v||^2).
__global__ void ref_residual_kernel(const float2 *__restrict__ v, const float2 *__restrict__ Wv,
                                    float2 *__restrict__ rout, Seg sg, int nblk, double2 *__restrict__ partial) {
    const int r = blockIdx.y;
    int64_t e0, e1;
    int local;
    const int s = chunk_system(sg, blockIdx.x, r, e0, e1, local);
    double q = 0, qv = 0;
    const int64_t n = sg.n;
#pragma unroll
    for (int t = 0; t < kEPT; ++t) {
        int64_t e = e0 + threadIdx.x + t * kDotThreads;
        if (e >= e1) continue;
        int64_t i = (int64_t)r * n + e;
        float2 a = v[i], b = Wv ? Wv[i] : make_float2(0.f, 0.f);
        double rx = (double)a.x - (double)b.x, ry = (double)a.y - (double)b.y;
        rout[i] = make_float2((float)rx, (float)ry);
        q += rx * rx + ry * ry;
        qv += (double)a.x * a.x + (double)a.y * a.y;
    }
    double2 tot = block_sum2(make_double2(q, qv));
    if (threadIdx.x == 0) partial[(int64_t)s * nblk + local] = tot;
}

__global__ void ref_accumulate_kernel(double2 *__restrict__ x64, const float2 *__restrict__ d, float2 *__restrict__ x32,
                                      int64_t total, int zero) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        double2 a = zero ? make_double2(0, 0) : x64[i];
        if (!zero) {
            a.x += d[i].x;
            a.y += d[i].y;
        }
        x64[i] = a;
        x32[i] = make_float2((float)a.x, (float)a.y);
    }
}

int vec_grid(int64_t n) {
    int64_t g = (n + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, 1024));
}

// The chunks of every scatterer's slice (host side).
struct Chunks {
    std::vector<int32_t> group, local, nchunk;
    std::vector<int64_t> start;
    int nblk = 1;
};

Chunks make_chunks(const ie_plan p) {
    Chunks c;
    c.nchunk.assign(p->ngroups, 0);
    for (int g = 0; g < p->ngroups; ++g) {
        const int64_t a = p->goff[g], b = p->goff[g + 1];
        int k = 0;
        for (int64_t e = a; e < b; e += kChunk, ++k) {
            c.group.push_back(g);
            c.start.push_back(e);
            c.local.push_back(k);
        }
        c.nchunk[g] = k;
        c.nblk = std::max(c.nblk, k);
    }
    if (c.group.empty()) {      // no unknowns at all: one empty chunk keeps the grids non-empty
        c.group.push_back(0);
        c.start.push_back(0);
        c.local.push_back(0);
    }
    return c;
}

Seg seg_of(const ie_solver s) {
    return Seg{s->chunk_group, s->chunk_start, s->chunk_local, s->goff, s->nchunk, s->G, s->n};
}

}  // namespace

void destroy_cached_solvers(ie_plan p) {
    for (auto &kv : p->solvers) ie_solver_destroy(kv.second);
    p->solvers.clear();
}

}  // namespace ie

using namespace ie;

namespace {

// A solver of `plan` for these options, created on first use and kept in the plan.
ie_status cached_solver(ie_plan p, int nrhs, const ie_solve_opts &o, ie_solver *out) {
    char key[160];
    snprintf(key, sizeof(key), "%d/%d/%d/%.17g/%d", nrhs, o.restart, o.max_iters, o.tol, o.prec);
    for (auto &kv : p->solvers)
        if (kv.first == key) {
            *out = kv.second;
            return IE_OK;
        }
    ie_solver s = nullptr;
    IE_TRY(ie_solver_create(p, nrhs, &o, &s));
    p->solvers.emplace_back(key, s);
    *out = s;
    return IE_OK;
}

ie_status salloc(ie_solver s, void **p, size_t bytes) {
    *p = nullptr;
    if (!bytes) return IE_OK;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("solver cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? IE_ERR_OOM : IE_ERR_CUDA;
    }
    s->allocs.push_back(*p);
    s->bytes += bytes;
    return IE_OK;
}
template <class T>
ie_status salloc_t(ie_solver s, T **p, size_t count) {
    return salloc(s, reinterpret_cast<void **>(p), count * sizeof(T));
}

size_t solver_bytes(int64_t n, int R, int G, int m, int C, int nblk, bool refine) {
    const int64_t S = (int64_t)R * G;
    size_t b = 0;
    b += (size_t)(m + 1) * R * n * sizeof(float2);           // V
    b += (size_t)2 * R * n * sizeof(float2);                 // W, Vcur
    b += (size_t)S * m * (m + 1) * sizeof(double2);          // H
    b += (size_t)S * m * (sizeof(double) + sizeof(double2)); // cs, sn
    b += (size_t)S * (m + 1) * sizeof(double2) * 2;          // g, hbuf
    b += (size_t)S * (m + 1) * nblk * sizeof(double2);       // partial
    b += (size_t)S * 2 * sizeof(double) + (6 + 5 * S + 2) * sizeof(int);   // bnorm, status, counters
    b += (size_t)C * (2 * sizeof(int32_t) + sizeof(int64_t)) + (size_t)(G + 1) * sizeof(int64_t) + G * sizeof(int32_t);
    if (refine) {      // refinement_buffers
        b += (size_t)R * n * (sizeof(double2) + 3 * sizeof(float2));
        b += (size_t)S * nblk * sizeof(double2);
    }
    return b;
}

void fill_defaults(ie_solve_opts *o) {
    o->restart = 50;
    o->max_iters = 1000;
    o->tol = 1e-6;
    o->prec = IE_PREC_FP32;
    o->refine = 0;
    o->refine_prec = IE_PREC_FP32;
    o->inner_tol = 1e-3;
    o->max_refine = 20;
}

Arnoldi arnoldi_of(const ie_solver s) {
    Arnoldi q;
    q.V = s->V, q.W = s->W, q.Vcur = s->Vcur;
    q.sg = seg_of(s);
    q.R = s->R, q.S = s->S, q.m = s->m, q.nblk = s->nblk;
    q.partial = s->partial, q.hbuf = s->hbuf, q.H = s->H, q.sn = s->sn, q.g = s->g;
    q.cs = s->cs, q.relres = s->relres;
    q.bnorm = s->bnorm;
    q.st = s->st, q.cnt = s->cnt;
    q.err = s->plan->d_err;
    q.tol = s->tol;
    q.max_iters = s->max_iters;
    return q;
}

// One Arnoldi iteration (product, CGS2, norm, Givens, scaling).  jarg = kDevJ takes
// the index from device memory (body of the WHILE node).
ie_status enqueue_iteration(ie_solver s, cudaStream_t st, int jarg) {
    const Arnoldi q = arnoldi_of(s);
    const dim3 cg(s->C, s->R);
    IE_TRY(apply(s->plan, IE_FULL, s->prec, s->Vcur, s->W, s->R, st, s->st));
    dots_kernel<<<cg, kDotThreads, 0, st>>>(q, jarg);
    update_dots_kernel<<<cg, kDotThreads, 0, st>>>(q, jarg);
    update_norm_kernel<<<cg, kDotThreads, 0, st>>>(q, jarg, s->hcond);
    scale_kernel<<<cg, kDotThreads, 0, st>>>(q, jarg == kDevJ ? kDevJ : jarg + 1);
    count_launches(3);   // the four kernels above (IE_CK_LAUNCH adds the last)
    IE_CK_LAUNCH();
    return IE_OK;
}

// Solution update x += V y and the restart: true residual, its norm, next cycle.
ie_status enqueue_end(ie_solver s, cudaStream_t st) {
    const int R = s->R, S = s->S, m = s->m;
    const Seg sg = seg_of(s);
    const dim3 cg(s->C, R);
    lsq_kernel<<<(S + 127) / 128, 128, 0, st>>>(s->H, s->g, s->hbuf, m, S, s->st);
    xupdate_kernel<<<cg, kDotThreads, 0, st>>>(s->V, s->x, sg, R, S, m, s->hbuf, s->st);
    count_launches(2);
    IE_TRY(apply(s->plan, IE_FULL, s->prec, s->x, s->W, R, st, s->st + 1));
    begin_cycle_kernel<<<cg, kDotThreads, 0, st>>>(arnoldi_of(s), s->v, s->x, 0, s->bnorm);
    scale_v0_kernel<<<cg, kDotThreads, 0, st>>>(s->V, s->Vcur, sg, S, m, s->hbuf, s->st);
    count_launches(1);   // begin_cycle (+ scale below)
    IE_CK_LAUNCH();
    return IE_OK;
}

int64_t count_kernel_nodes(cudaGraph_t graph) {
    size_t nn = 0;
    if (cudaGraphGetNodes(graph, nullptr, &nn) != cudaSuccess) return 0;
    std::vector<cudaGraphNode_t> nodes(nn);
    if (nn && cudaGraphGetNodes(graph, nodes.data(), &nn) != cudaSuccess) return 0;
    int64_t k = 0;
    for (auto nd : nodes) {
        cudaGraphNodeType t;
        if (cudaGraphNodeGetType(nd, &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) k++;
    }
    return k;
}

// One restart cycle as a graph: a WHILE node whose body is one Arnoldi iteration
// (the Givens kernel sets the condition from the per-system flags), then the end of
// the cycle.  Skipped iterations cost nothing and the cycle needs no host sync.
ie_status build_while_graph(ie_solver s, cudaGraph_t *out) {
    cudaGraph_t g = nullptr;
    IE_CK(cudaGraphCreate(&g, 0));
    auto fail = [&](cudaError_t e, const char *what) {
        cudaGetLastError();
        cudaGraphDestroy(g);
        set_error("%s: %s", what, cudaGetErrorString(e));
        return IE_ERR_CUDA;
    };
    cudaError_t e = cudaGraphConditionalHandleCreate(&s->hcond, g, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return fail(e, "cudaGraphConditionalHandleCreate");
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = s->hcond;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t wnode;
    e = cudaGraphAddNode(&wnode, g, nullptr, nullptr, 0, &cp);
    if (e != cudaSuccess) return fail(e, "cudaGraphAddNode(while)");
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    e = cudaStreamBeginCaptureToGraph(s->cap, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return fail(e, "capture body");
    capture_begin();
    ie_status st1 = enqueue_iteration(s, s->cap, kDevJ);
    capture_end();
    cudaGraph_t tmp = nullptr;
    e = cudaStreamEndCapture(s->cap, &tmp);
    if (st1 != IE_OK) {
        cudaGraphDestroy(g);
        return st1;
    }
    if (e != cudaSuccess) return fail(e, "end capture body");
    s->body_kernels = count_kernel_nodes(body);
    e = cudaStreamBeginCaptureToGraph(s->cap, g, &wnode, nullptr, 1, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return fail(e, "capture end");
    capture_begin();
    ie_status st2 = enqueue_end(s, s->cap);
    capture_end();
    e = cudaStreamEndCapture(s->cap, &tmp);
    if (st2 != IE_OK) {
        cudaGraphDestroy(g);
        return st2;
    }
    if (e != cudaSuccess) return fail(e, "end capture end");
    s->end_kernels = count_kernel_nodes(g);
    *out = g;
    return IE_OK;
}

// Fallback: the m iterations unrolled with explicit indices (every kernel gated).
ie_status build_unrolled_graph(ie_solver s, cudaGraph_t *out) {
    s->hcond = 0;
    IE_CK(cudaStreamBeginCapture(s->cap, cudaStreamCaptureModeThreadLocal));
    capture_begin();
    ie_status e = IE_OK;
    for (int j = 0; j < s->m && e == IE_OK; ++j) e = enqueue_iteration(s, s->cap, j);
    if (e == IE_OK) e = enqueue_end(s, s->cap);
    capture_end();
    cudaGraph_t graph = nullptr;
    cudaError_t ce = cudaStreamEndCapture(s->cap, &graph);
    if (e != IE_OK) {
        if (graph) cudaGraphDestroy(graph);
        return e;
    }
    IE_CK(ce);
    s->body_kernels = 0;
    s->end_kernels = count_kernel_nodes(graph);
    *out = graph;
    return IE_OK;
}

// Status and counts from the pinned mirror (valid once the solver's event has completed).
void read_info_mirror(ie_solver s, ie_solve_info *info, int *done) {
    const int S = s->S;
    const int *st = s->h_st;
    if (done) *done = st[1] == 0;
    if (!info) return;
    int it = 0;
    double rr = 0;
    bool conv = true;
    for (int q = 0; q < S; ++q) {
        it = std::max(it, st[2 + 3 * S + q]);
        rr = std::max(rr, s->h_rel[q]);
        if (s->h_rel[q] > s->tol) conv = false;
    }
    info->iterations = it;
    info->relres = rr;
    info->converged = conv ? 1 : 0;
    const int64_t body = st[3 + 4 * S];
    info->matvecs = (int)(s->use_while ? body + s->cycles_run : (int64_t)s->cycles_run * s->matvecs_per_cycle);
    if (s->use_while && body > s->body_runs_seen) {
        count_launches((body - s->body_runs_seen) * s->body_kernels);
        s->body_runs_seen = body;
    }
}

// st and, on an 8-byte boundary behind it, relres: one device block and its pinned mirror.
size_t rel_offset(int S) { return ((size_t)st_ints(S) * sizeof(int) + 7) / 8 * 8; }
size_t status_bytes(int S) { return rel_offset(S) + S * sizeof(double); }

// Enqueue the copy of the status into the pinned mirror and record the solver's event.
ie_status mirror_status(ie_solver s, cudaStream_t st) {
    IE_CK(cudaMemcpyAsync(s->h_st, s->st, status_bytes(s->S), cudaMemcpyDeviceToHost, st));
    IE_CK(cudaEventRecord(s->ev, st));
    return IE_OK;
}

// Device and pinned buffers of the outer refinement, kept with the (plan's) solver: a call
// then allocates nothing, and the captured cycle's pointers stay the same from call to call.
ie_status refinement_buffers(ie_solver s) {
    if (s->h_part) return IE_OK;
    std::lock_guard<std::recursive_mutex> lock(device_mutex());
    const size_t total = (size_t)s->R * s->n, np = (size_t)s->S * s->nblk;
    if (!s->x64) IE_TRY(salloc_t(s, &s->x64, total));
    if (!s->rv) IE_TRY(salloc_t(s, &s->rv, total));
    if (!s->rd) IE_TRY(salloc_t(s, &s->rd, total));
    if (!s->rw) IE_TRY(salloc_t(s, &s->rw, total));
    if (!s->rpart) IE_TRY(salloc_t(s, &s->rpart, np));
    void *h = nullptr;
    if (cudaMallocHost(&h, np * sizeof(double2)) != cudaSuccess) {
        cudaGetLastError();
        return set_error("pinned refinement sums allocation failed"), IE_ERR_OOM;
    }
    s->h_part = static_cast<double2 *>(h);
    return IE_OK;
}

// Cycles until every system is done (or the cycle cap), synchronising once per cycle.
ie_status run_cycles(ie_solver s, const ie_solve_opts &o, void *stream, ie_solve_info *inf) {
    cudaStream_t st = (cudaStream_t)stream;
    int done = 0;
    const int max_cycles = (o.max_iters + o.restart - 1) / o.restart + 2;
    for (int cyc = 0; !done && cyc < max_cycles; ++cyc) {
        IE_TRY(ie_solver_advance(s, 1, stream));
        IE_CK(cudaStreamSynchronize(st));
        read_info_mirror(s, inf, &done);     // the advance copied the status to the host
    }
    return IE_OK;
}

}  // namespace

extern "C" {

void ie_solve_opts_default(ie_solve_opts *o) {
    if (o) fill_defaults(o);
}

ie_status ie_solver_footprint(ie_plan p, int nrhs, const ie_solve_opts *opts, size_t *bytes) {
    if (!p || !bytes) return set_error("null argument"), IE_ERR_INVALID;
    ie_solve_opts o;
    fill_defaults(&o);
    if (opts) o = *opts;
    Chunks c = make_chunks(p);
    *bytes = solver_bytes(p->n, nrhs, p->ngroups, o.restart, (int)c.group.size(), c.nblk, o.refine != 0);
    return IE_OK;
}

ie_status ie_solver_create(ie_plan p, int nrhs, const ie_solve_opts *opts, ie_solver *out) {
    if (!p || !out) return set_error("null argument"), IE_ERR_INVALID;
    std::lock_guard<std::recursive_mutex> lock(device_mutex());
    *out = nullptr;
    ie_solve_opts o;
    fill_defaults(&o);
    if (opts) o = *opts;
    if (nrhs < 1 || nrhs > p->max_rhs || nrhs > 64) return set_error("bad nrhs %d", nrhs), IE_ERR_INVALID;
    if (o.restart < 1 || o.restart > 64) return set_error("restart must be in [1, 64]"), IE_ERR_INVALID;
    if (o.refine) return set_error("solver objects do not refine; use ie_solve"), IE_ERR_INVALID;
    if ((int64_t)nrhs * p->ngroups > kMaxSystems)
        return set_error("%d right-hand sides x %d scatterers exceed %d systems", nrhs, p->ngroups, kMaxSystems),
               IE_ERR_INVALID;
    if (!(p->prec_mask & IE_PRECMASK(o.prec))) return set_error("precision not in plan"), IE_ERR_UNSUPPORTED;
    ie_solver s = new ie_solver_s();
    auto fail = [&](ie_status st) {
        ie_solver_destroy(s);
        return st;
    };
    s->plan = p;
    s->R = nrhs;
    s->G = p->ngroups;
    s->S = nrhs * p->ngroups;
    s->m = o.restart;
    s->max_iters = o.max_iters;
    s->tol = o.tol;
    s->prec = o.prec;
    s->n = p->n;
    Chunks c = make_chunks(p);
    s->C = (int)c.group.size();
    s->nblk = c.nblk;
    const int R = nrhs, S = s->S, m = o.restart;
    ie_status e;
#define SA(ptr, cnt)                                   \
    do {                                               \
        e = salloc_t(s, &(ptr), (size_t)(cnt));        \
        if (e != IE_OK) return fail(e);                \
    } while (0)
    SA(s->chunk_group, s->C);
    SA(s->chunk_start, s->C);
    SA(s->chunk_local, s->C);
    SA(s->goff, s->G + 1);
    SA(s->nchunk, s->G);
    SA(s->V, (size_t)(m + 1) * R * s->n);
    SA(s->W, (size_t)R * s->n);
    SA(s->Vcur, (size_t)R * s->n);
    SA(s->H, (size_t)S * m * (m + 1));
    SA(s->cs, (size_t)S * m);
    SA(s->sn, (size_t)S * m);
    SA(s->g, (size_t)S * (m + 1));
    SA(s->hbuf, (size_t)S * (m + 1));
    SA(s->partial, (size_t)S * (m + 1) * s->nblk);
    SA(s->bnorm, S);
    SA(s->cnt, S + 1);
    {
        char *block = nullptr;
        SA(block, status_bytes(S));
        s->st = reinterpret_cast<int *>(block);
        s->relres = reinterpret_cast<double *>(block + rel_offset(S));
    }
#undef SA
    if (cudaMemcpy(s->chunk_group, c.group.data(), s->C * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->chunk_start, c.start.data(), s->C * sizeof(int64_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->chunk_local, c.local.data(), s->C * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->goff, p->goff.data(), (s->G + 1) * sizeof(int64_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->nchunk, c.nchunk.data(), s->G * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(s->st, 0, status_bytes(S)) != cudaSuccess ||
        cudaMemset(s->cnt, 0, (S + 1) * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        set_error("solver set-up copies failed");
        return fail(IE_ERR_CUDA);
    }
    // work lists must exist before graph capture (they allocate); the convolution has none
    WorkList *wl = nullptr;
    e = conv_full(p, o.prec) ? IE_OK : work_list_for(p, o.prec, R, &wl);
    if (e != IE_OK) return fail(e);
    if (cudaStreamCreateWithFlags(&s->cap, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&s->ev, cudaEventDisableTiming) != cudaSuccess) {
        set_error("stream/event creation failed");
        return fail(IE_ERR_CUDA);
    }
    {
        void *h = nullptr;
        if (cudaMallocHost(&h, status_bytes(S)) != cudaSuccess) {
            cudaGetLastError();
            set_error("pinned status mirror allocation failed");
            return fail(IE_ERR_OOM);
        }
        s->h_st = static_cast<int *>(h);
        s->h_rel = reinterpret_cast<double *>(static_cast<char *>(h) + rel_offset(S));
        memset(h, 0, status_bytes(S));
    }
    s->matvecs_per_cycle = m + 1;
    *out = s;
    return IE_OK;
}

ie_status ie_solver_destroy(ie_solver s) {
    if (!s) return IE_OK;
    std::lock_guard<std::recursive_mutex> lock(device_mutex());
    cudaDeviceSynchronize();
    if (s->exec) cudaGraphExecDestroy(s->exec);
    if (s->cap) cudaStreamDestroy(s->cap);
    if (s->ev) cudaEventDestroy(s->ev);
    for (void *q : s->allocs) cudaFree(q);
    if (s->h_st) cudaFreeHost(s->h_st);
    if (s->h_part) cudaFreeHost(s->h_part);
    delete s;
    return IE_OK;
}

ie_status ie_solver_start(ie_solver s, const void *v, void *c, void *stream) {
    if (!s || !v || !c) return set_error("null argument"), IE_ERR_INVALID;
    cudaStream_t st = (cudaStream_t)stream;
    s->v = (const float2 *)v;
    s->x = (float2 *)c;
    s->cycles_run = 0;
    const int R = s->R, S = s->S, m = s->m;
    const Seg sg = seg_of(s);
    const dim3 cg(s->C, R);
    IE_CK(cudaMemsetAsync(s->st, 0, st_ints(S) * sizeof(int), st));
    s->body_runs_seen = 0;
    begin_cycle_kernel<<<cg, kDotThreads, 0, st>>>(arnoldi_of(s), s->v, s->x, 1, s->bnorm);
    scale_v0_kernel<<<cg, kDotThreads, 0, st>>>(s->V, s->Vcur, sg, S, m, s->hbuf, s->st);
    count_launches(1);
    IE_CK_LAUNCH();
    IE_TRY(mirror_status(s, st));
    // the captured cycle reads v and x through fixed pointers: recapture if they moved
    if (s->exec && (s->cap_v != s->v || s->cap_x != s->x)) {
        cudaGraphExecDestroy(s->exec);
        s->exec = nullptr;
    }
    return IE_OK;
}

ie_status ie_solver_advance(ie_solver s, int cycles, void *stream) {
    ie::NvtxRange nvtx_range("ie_solver_advance");
    if (!s || cycles < 0) return set_error("bad argument"), IE_ERR_INVALID;
    cudaStream_t st = (cudaStream_t)stream;
    for (int c = 0; c < cycles; ++c) {
        if (!s->exec) {
            std::lock_guard<std::recursive_mutex> lock(device_mutex());
            // build the cycle graph on the private stream, ordered after `st`
            IE_CK(cudaEventRecord(s->ev, st));
            IE_CK(cudaStreamWaitEvent(s->cap, s->ev, 0));
            cudaGraph_t graph = nullptr;
            s->use_while = build_while_graph(s, &graph) == IE_OK;
            if (!s->use_while) IE_TRY(build_unrolled_graph(s, &graph));
            cudaError_t ie_ = cudaGraphInstantiate(&s->exec, graph, 0);
            cudaGraphDestroy(graph);
            IE_CK(ie_);
            s->cap_v = s->v;
            s->cap_x = s->x;
        }
        IE_CK(cudaGraphLaunch(s->exec, st));
        count_launches(s->end_kernels);
        s->cycles_run++;
    }
    return mirror_status(s, st);
}

ie_status ie_solver_poll(ie_solver s, int *done, ie_solve_info *info) {
    if (!s || !done) return set_error("null argument"), IE_ERR_INVALID;
    cudaError_t q = cudaEventQuery(s->ev);
    if (q == cudaErrorNotReady) {
        *done = 0;
        return IE_OK;
    }
    IE_CK(q);
    read_info_mirror(s, info, done);
    return IE_OK;
}

ie_status ie_solver_state(ie_solver s, int *state, ie_solve_info *info) {
    if (!s || !state) return set_error("null argument"), IE_ERR_INVALID;
    cudaError_t q = cudaEventQuery(s->ev);
    if (q == cudaErrorNotReady) {
        *state = IE_SOLVER_BUSY;
        return IE_OK;
    }
    IE_CK(q);
    int done = 0;
    read_info_mirror(s, info, &done);
    *state = done ? IE_SOLVER_DONE : IE_SOLVER_IDLE;
    return IE_OK;
}

ie_status ie_solve(ie_plan p, const void *v, void *c, int nrhs, const ie_solve_opts *opts, ie_solve_info *info,
                   void *stream) {
    ie::NvtxRange nvtx_range("ie_solve");
    auto t0 = std::chrono::steady_clock::now();
    if (!p || !v || !c) return set_error("null argument"), IE_ERR_INVALID;
    ie_solve_opts o;
    fill_defaults(&o);
    if (opts) o = *opts;
    cudaStream_t st = (cudaStream_t)stream;
    ie_solve_info inf{};
    ie_status result = IE_OK;
    // whether the solver's status copy shows every product's error word so far
    bool seen = false, clean = true;
    auto look = [&](ie_solver s) {
        seen = true;
        clean = clean && s->h_st[4 + 4 * s->S] == 0;
    };
    if (!o.refine) {
        ie_solver s = nullptr;
        IE_TRY(cached_solver(p, nrhs, o, &s));
        IE_TRY(ie_solver_start(s, v, c, stream));
        IE_TRY(run_cycles(s, o, stream, &inf));
        look(s);
        result = inf.converged ? IE_OK : IE_ERR_NOT_CONVERGED;
    } else {
        // outer refinement: x64 += GMRES_prec(r), r = v - Z_refine(x) in FP64, per system
        if (!(p->prec_mask & IE_PRECMASK(o.refine_prec)) || !(p->prec_mask & IE_PRECMASK(o.prec)))
            return set_error("refinement precisions not in plan"), IE_ERR_UNSUPPORTED;
        ie_solve_opts io = o;
        io.refine = 0;
        io.tol = o.inner_tol;
        ie_solver s = nullptr;
        IE_TRY(cached_solver(p, nrhs, io, &s));
        const int64_t total = (int64_t)nrhs * p->n;
        const int S = s->S, nblk = s->nblk, G = s->G;
        const Seg sg = seg_of(s);
        IE_TRY(refinement_buffers(s));
        double2 *const x64 = s->x64, *const part = s->rpart, *const hp = s->h_part;
        float2 *const rv = s->rv, *const d = s->rd, *const Wz = s->rw;
        const size_t nhp = (size_t)S * nblk;
        IE_CK(cudaMemsetAsync(part, 0, nhp * sizeof(double2), st));
        ref_accumulate_kernel<<<vec_grid(total), 256, 0, st>>>(x64, nullptr, (float2 *)c, total, 1);
        count_launches(1);
        std::vector<int> nch(G);
        for (int g = 0; g < G; ++g) nch[g] = (int)((p->goff[g + 1] - p->goff[g] + kChunk - 1) / kChunk);
        int outer = 0, inner_iters = 0, mv = 0;
        double worst = 1;
        ie_status e = IE_OK;
        bool reuse = false;     // the inner solver's last product is Z c in refine_prec
        while (e == IE_OK) {
            // r = v - Z x  (FP64 difference of the product); x = 0 on the first step, so r = v
            const float2 *Zc = nullptr;
            if (reuse) {
                Zc = s->W;
            } else if (outer > 0) {
                e = apply(p, IE_FULL, o.refine_prec, (const float2 *)c, Wz, nrhs, st);
                seen = false;
                mv++;
                if (e != IE_OK) break;
                Zc = Wz;
            }
            ref_residual_kernel<<<dim3(s->C, nrhs), kDotThreads, 0, st>>>((const float2 *)v, Zc, rv, sg, nblk, part);
            count_launches(1);
            if (cudaMemcpyAsync(hp, part, nhp * sizeof(double2), cudaMemcpyDeviceToHost, st) !=
                    cudaSuccess ||
                cudaStreamSynchronize(st) != cudaSuccess) {
                set_error("refinement residual copy failed");
                e = IE_ERR_CUDA;
                break;
            }
            worst = 0;
            for (int q = 0; q < S; ++q) {
                double rs = 0, vs = 0;
                for (int b = 0; b < nch[q % G]; ++b) rs += hp[(size_t)q * nblk + b].x, vs += hp[(size_t)q * nblk + b].y;
                worst = std::max(worst, vs > 0 ? std::sqrt(rs / vs) : 0.0);
            }
            if (worst <= o.tol || outer >= o.max_refine || inner_iters >= o.max_iters) break;
            // inner solve Z d = r
            e = ie_solver_start(s, rv, d, stream);
            ie_solve_info ii{};
            if (e == IE_OK) e = run_cycles(s, io, stream, &ii);
            if (e != IE_OK) break;
            look(s);
            inner_iters += ii.iterations;
            mv += ii.matvecs;
            ref_accumulate_kernel<<<vec_grid(total), 256, 0, st>>>(x64, d, (float2 *)c, total, 0);
            count_launches(1);
            // After the first inner solve x = 0 + d exactly (c = d), and the inner solver's
            // restart product W = Z d was taken with the last update of d: when it used the
            // refinement's precision, the next residual reuses it instead of a new product.
            reuse = outer == 0 && ii.iterations > 0 && io.prec == o.refine_prec;
            outer++;
        }
        if (e != IE_OK) return e;
        inf.iterations = inner_iters;
        inf.matvecs = mv;
        inf.refinements = outer;
        inf.relres = worst;
        inf.converged = worst <= o.tol;
        result = inf.converged ? IE_OK : IE_ERR_NOT_CONVERGED;
    }
    inf.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (info) *info = inf;
    // a translation that gave up a wait voids the solve; the status copy carries the error word
    // of every product before it, so another round trip is only needed without one
    if (!seen || !clean) IE_TRY(take_device_error(p, st));
    return result;
}

}  // extern "C"

// Mapping construction of §2.1 (eq. 9-11): the rows of P_b for subdomain basis
// functions made of point dipoles.  The 192 uniform dipoles of a box radiate A
// (3 N_s x 192) at N_s Fibonacci samples on a sphere S about the box centre; a
// function radiates B_f there (eq. 4); eq. 11 takes C_f = A^+ B_f, row f of P_b.
//
// A is the same for every box, so A^+ is formed once: a Householder QR of A by one CTA per
// column with the columns of Q_1 formed from the reflectors, then one warp per sample row
// back-substitutes with R, which gives column i of A^+ = R^-1 Q_1^H.  With a Tikhonov weight the factorised
// matrix is [A; lambda I] (lambda = t ||A||_F) and the first 3 N_s columns of its
// pseudo-inverse are (A^H A + lambda^2 I)^-1 A^H.  The per-function work (fields on S,
// the product with A^+, the residual on S) is one CTA per 8 functions.  All FP64:
// A's condition number is about 1e7, so FP32 would lose the fit.
#include "ie_internal.h"

#include <algorithm>
#include <cmath>
#include <vector>

namespace ie {
namespace {

constexpr int kMinSamples = 64;                   // 3 N_s >= 192: full column rank possible
constexpr int kMaxSamples = 256;
constexpr int kFunPerCta = 8;
constexpr int kMapThreads = 2 * kNU;
constexpr int64_t kMapChunk = int64_t(1) << 16;   // functions per device pass

struct Sphere {
    double k, eta, a, radius;   // radius of S (absolute)
    int ns;                     // samples on S
};

__device__ inline void cmac(double2 &acc, double2 a, double2 b) {   // acc += a b
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}
// Sample l of the spherical Fibonacci lattice on S: polar angle arccos(1 - (2l+1)/N_s),
// azimuth 2 pi l / golden ratio.
__device__ inline void sample_point(const Sphere &s, int l, double r[3]) {
    constexpr double kPi = 3.14159265358979323846;
    const double golden = 0.5 + 0.5 * sqrt(5.0);
    double z = 1.0 - (2.0 * l + 1.0) / s.ns;
    double st = sqrt((1.0 - z) * (1.0 + z));
    double sa, ca;
    sincos(2.0 * kPi * l / golden, &sa, &ca);
    r[0] = s.radius * st * ca;
    r[1] = s.radius * st * sa;
    r[2] = s.radius * z;
}

// A (column-major, 3 N_s rows): entry (3l + alpha, 3j + beta) = D_{alpha beta}(r_l - s_j),
// s_j the cell-centred lattice site j of a box centred at the origin.  One thread per
// (sample, site).  Written into the factorised matrix (leading dimension lda >= 3 N_s)
// and into A0 (leading dimension 3 N_s), kept for the residuals.
__global__ void sample_matrix_kernel(Sphere s, double2 *__restrict__ A, int lda, double2 *__restrict__ A0) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= s.ns * kSites) return;
    int l = t % s.ns, j = t / s.ns;
    double r[3];
    sample_point(s, l, r);
    const double h = s.a / kLattice;
    double q[3] = {h * ((j & 3) + 0.5) - 0.5 * s.a, h * (((j >> 2) & 3) + 0.5) - 0.5 * s.a,
                   h * ((j >> 4) + 0.5) - 0.5 * s.a};
    double2 D[9];
    dyad_fp64(s.k, s.eta, r[0] - q[0], r[1] - q[1], r[2] - q[2], D);
    const size_t m = 3 * (size_t)s.ns;
#pragma unroll
    for (int al = 0; al < 3; ++al)
#pragma unroll
        for (int be = 0; be < 3; ++be) {
            const size_t row = 3 * (size_t)l + al, col = 3 * (size_t)j + be;
            A[row + (size_t)lda * col] = D[3 * al + be];
            A0[row + m * col] = D[3 * al + be];
        }
}

// Pseudo-inverse, first part: the Householder QR of A (m x 192, column-major, m <= 960), one
// CTA per column, the columns in registers.  Step j maps column j below the diagonal onto
// alpha e_j with H_j = I - tau_j v_j v_j^H, alpha = -e^{i arg x0} ||x||, v_j = x - alpha e_j
// (V, rows j..m-1), tau_j = 2 / ||v_j||^2; R goes to the upper triangle of A.  CTA j publishes
// v_j and raises flag[j]; the later CTAs apply it, CTA j + 1 then publishes at once.  Then
// each CTA forms its column of Q_1 = H_0 .. H_191 [I; 0] (conjugated rows, Y[i][c], i <
// m_data), needing only the published vectors.  *status = 1 if a column is zero (rank
// deficient), 2 if a wait gave up.
// tikhonov > 0: rows m_data .. m_data+191 are lambda I, lambda = tikhonov ||A[0 .. m_data)||_F.
// Bound by the chain of 192 steps, and a step by FP64 issue (64 cycles per warp instruction and
// SM quarter): four warps per CTA, one per quarter, no row outside [j, m), re and im reduced
// in one shuffle tree.  m = 576: 2.5 ms; all columns in one CTA took 37 ms.
constexpr int kQrThreads = 128, kQrWarps = kQrThreads / 32, kQrRows = 8;
static_assert(kQrRows * kQrThreads >= 3 * kMaxSamples + kNU, "columns in registers");
constexpr long long kQrWaitCycles = 1ll << 31;      // bounded wait, ~1 s

// Sum over the block, the result in every thread.  The first exchange leaves re in the lower
// and im in the upper half-warp.
__device__ inline double2 block_sum(double2 v, double (*red)[2][kQrWarps], int &slot) {
    const int lane = threadIdx.x & 31, hi = lane >> 4;
    double x = (hi ? v.y : v.x) + __shfl_xor_sync(0xffffffffu, hi ? v.x : v.y, 16);
    for (int o = 8; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((lane & 15) == 0) red[slot][hi][threadIdx.x >> 5] = x;
    __syncthreads();
    const double *r = red[slot][0], *i = red[slot][1];
    slot ^= 1;          // two buffers: one barrier per sum
    return make_double2((r[0] + r[1]) + (r[2] + r[3]), (i[0] + i[1]) + (i[2] + i[3]));
}
static_assert(kQrWarps == 4, "four partial sums");

__global__ void __launch_bounds__(kQrThreads) qr_kernel(double2 *__restrict__ A, const double2 *__restrict__ A0, int m,
                                                        int m_data, double tikhonov, double2 *V, double *tau, int *flag,
                                                        double2 *__restrict__ Y, int *__restrict__ status) {
    __shared__ double red[2][2][kQrWarps];
    __shared__ double2 s_x0, s_ph;
    __shared__ double s_ax0;
    __shared__ int s_ok;
    const int tid = threadIdx.x, c = blockIdx.x, w0 = tid & ~31;
    int slot = 0;
    double lambda = 0.0;
    if (tikhonov > 0.0) {       // every CTA sums ||A||_F itself, in the same order, from the copy
        double2 ss = make_double2(0.0, 0.0);    // (R already replaces columns of A elsewhere)
        for (int i = tid; i < m_data * kNU; i += kQrThreads) {
            const double2 x = A0[i];
            ss.x = fma(x.x, x.x, ss.x), ss.y = fma(x.y, x.y, ss.y);
        }
        ss = block_sum(ss, red, slot);
        lambda = tikhonov * sqrt(ss.x + ss.y);
    }
    double2 x[kQrRows];
#pragma unroll
    for (int t = 0; t < kQrRows; ++t) {
        const int i = tid + t * kQrThreads;
        x[t] = i < m_data ? A[i + (size_t)m * c] : make_double2(i < m && i - m_data == c ? lambda : 0.0, 0.0);
    }
    // rows of this warp's chunk t that a step over rows [j, m) touches
    auto live = [&](int t, int j) { return w0 + t * kQrThreads < m && w0 + t * kQrThreads + 31 >= j; };
    double2 v[kQrRows];
    auto fetch = [&](int j) {
#pragma unroll
        for (int t = 0; t < kQrRows; ++t) {
            const int i = tid + t * kQrThreads;
            v[t] = live(t, j) && i < m ? __ldcg(V + i + (size_t)m * j) : make_double2(0.0, 0.0);
        }
    };
    // x <- H_j x, v = v_j (zero above row j)
    auto reflect = [&](int j, double tj) {
        double2 d = make_double2(0.0, 0.0);
#pragma unroll
        for (int t = 0; t < kQrRows; ++t)
            if (live(t, j)) {
                d.x = fma(v[t].x, x[t].x, fma(v[t].y, x[t].y, d.x));
                d.y = fma(v[t].x, x[t].y, fma(-v[t].y, x[t].x, d.y));
            }
        d = block_sum(d, red, slot);
        const double fx = tj * d.x, fy = tj * d.y;
#pragma unroll
        for (int t = 0; t < kQrRows; ++t)
            if (live(t, j)) {
                x[t].x = fma(-fx, v[t].x, fma(fy, v[t].y, x[t].x));
                x[t].y = fma(-fx, v[t].y, fma(-fy, v[t].x, x[t].y));
            }
    };
    for (int j = 0; j < c; ++j) {
        if (tid == 0) {
            const long long t0 = clock64();
            int f = 0;
            while (!f && clock64() - t0 < kQrWaitCycles)
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(f) : "l"(flag + j) : "memory");
            s_ok = f;
        }
        __syncthreads();
        if (!s_ok) {            // the same in every thread
            if (tid == 0) atomicMax(status, 2);
            return;
        }
        fetch(j);
        reflect(j, __ldcg(tau + j));
    }
    double tc;
    {   // the reflector of the own column
        double2 ss = make_double2(0.0, 0.0);
#pragma unroll
        for (int t = 0; t < kQrRows; ++t) {
            const int i = tid + t * kQrThreads;
            if (i == c) s_x0 = x[t];
            if (live(t, c) && i >= c) ss.x = fma(x[t].x, x[t].x, ss.x), ss.y = fma(x[t].y, x[t].y, ss.y);
        }
        __syncthreads();
        const double2 x0 = s_x0;
        if (w0 == 32 * (kQrWarps - 1)) {       // beside the other warps' sums
            const double ax = hypot(x0.x, x0.y);
            if (tid == w0) {
                s_ax0 = ax;
                s_ph = ax > 0.0 ? make_double2(x0.x / ax, x0.y / ax) : make_double2(1.0, 0.0);
            }
        }
        ss = block_sum(ss, red, slot);
        const double xn = sqrt(ss.x + ss.y), ax0 = s_ax0;
        const double2 ph = s_ph;
        tc = xn > 0.0 ? 1.0 / (xn * (xn + ax0)) : 0.0;             // ||v||^2 = 2 xn (xn + |x0|)
#pragma unroll
        for (int t = 0; t < kQrRows; ++t) {
            const int i = tid + t * kQrThreads;
            v[t] = i > c ? x[t] : make_double2(0.0, 0.0);
            if (i == c && xn > 0.0) v[t] = make_double2(ph.x * (ax0 + xn), ph.y * (ax0 + xn));
            if (i < m) V[i + (size_t)m * c] = v[t];
            if (i <= c)         // column c of R, R_cc = alpha
                A[i + (size_t)m * c] = i < c ? x[t] : make_double2(-ph.x * xn, -ph.y * xn);
        }
        if (tid == 0) {
            tau[c] = tc;
            if (xn == 0.0) atomicMax(status, 1);
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) asm volatile("st.release.gpu.global.s32 [%0], 1;" ::"l"(flag + c) : "memory");
    }
    // column c of Q_1: H_c .. H_0 applied to e_c (H_j with j > c leaves it as it is)
#pragma unroll
    for (int t = 0; t < kQrRows; ++t) x[t] = make_double2(tid + t * kQrThreads == c ? 1.0 : 0.0, 0.0);
    reflect(c, tc);
    for (int j = c - 1; j >= 0; --j) {
        fetch(j);
        reflect(j, __ldcg(tau + j));
    }
#pragma unroll
    for (int t = 0; t < kQrRows; ++t) {
        const int i = tid + t * kQrThreads;
        if (i < m_data) Y[(size_t)i * kNU + c] = make_double2(x[t].x, -x[t].y);
    }
}

// Second part: column i of A^+ = R^-1 Q_1^H (row i of Apinv, [m_data][192]) from row i of
// conj(Q_1), in place, by back substitution.  One warp per row, six unknowns per lane; the
// next column of R is in flight during a step.
__global__ void __launch_bounds__(32) pinv_solve_kernel(const double2 *__restrict__ R, int m, double2 *__restrict__ Y) {
    const int lane = threadIdx.x;
    double2 *row = Y + (size_t)blockIdx.x * kNU;
    double2 y[kNU / 32], r[kNU / 32];
#pragma unroll
    for (int t = 0; t < kNU / 32; ++t) y[t] = row[lane + 32 * t];
    auto fetch = [&](int c) {
#pragma unroll
        for (int t = 0; t < kNU / 32; ++t)
            r[t] = lane + 32 * t <= c ? R[lane + 32 * t + (size_t)m * c] : make_double2(0.0, 0.0);
    };
    fetch(kNU - 1);
#pragma unroll
    for (int tc = kNU / 32 - 1; tc >= 0; --tc)
        for (int lc = 31; lc >= 0; --lc) {
            const int c = 32 * tc + lc;
            double2 cur[kNU / 32];
#pragma unroll
            for (int t = 0; t < kNU / 32; ++t) cur[t] = r[t];
            if (c > 0) fetch(c - 1);
            const double2 yr = make_double2(__shfl_sync(0xffffffffu, y[tc].x, lc), __shfl_sync(0xffffffffu, y[tc].y, lc));
            const double2 rr = make_double2(__shfl_sync(0xffffffffu, cur[tc].x, lc),
                                            __shfl_sync(0xffffffffu, cur[tc].y, lc));
            const double den = rr.x * rr.x + rr.y * rr.y;
            const double2 x = make_double2((yr.x * rr.x + yr.y * rr.y) / den, (yr.y * rr.x - yr.x * rr.y) / den);
#pragma unroll
            for (int t = 0; t <= tc; ++t) {
                const int i = lane + 32 * t;
                if (i < c) {
                    y[t].x = fma(-cur[t].x, x.x, fma(cur[t].y, x.y, y[t].x));
                    y[t].y = fma(-cur[t].x, x.y, fma(-cur[t].y, x.x, y[t].y));
                } else if (i == c) {
                    y[t] = x;
                }
            }
        }
#pragma unroll
    for (int t = 0; t < kNU / 32; ++t) row[lane + 32 * t] = y[t];
}

struct MapArgs {
    Sphere s;
    int64_t n_fun;
    const int64_t *off;       // n_fun + 1, rebased to this chunk's dipoles
    const double *pos;        // [dipole][3]
    const double2 *mom;       // [dipole][3]
    const double2 *Apinv;     // [m][192]
    const double2 *A0;        // [192][m] (column-major A)
    double2 *P;               // [n_fun][192]
    double *res;              // [n_fun] or null
};

// Eight functions per CTA: their fields on S (eq. 4 summed over the point dipoles),
// C_f = A^+ B_f (eq. 11), and ||A C_f - B_f|| / ||B_f||.  FP64 rate bound: 192 x 384 x 2 complex
// multiply-adds per function, four FMAs each.
__global__ void __launch_bounds__(kMapThreads) map_kernel(MapArgs g) {
    extern __shared__ double2 sm[];
    __shared__ double red[2][kFunPerCta][kMapThreads / 32];
    const int m = 3 * g.s.ns;
    double2 *B = sm;                        // [kFunPerCta][m]
    double2 *C = sm + kFunPerCta * m;       // [kFunPerCta][192]
    const int64_t f0 = (int64_t)blockIdx.x * kFunPerCta;
    for (int idx = threadIdx.x; idx < kFunPerCta * g.s.ns; idx += blockDim.x) {
        const int t = idx / g.s.ns, l = idx % g.s.ns;
        const int64_t f = f0 + t;
        double2 e[3] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
        if (f < g.n_fun) {
            double r[3];
            sample_point(g.s, l, r);
            for (int64_t d = g.off[f]; d < g.off[f + 1]; ++d) {
                double2 D[9];
                dyad_fp64(g.s.k, g.s.eta, r[0] - g.pos[3 * d], r[1] - g.pos[3 * d + 1], r[2] - g.pos[3 * d + 2], D);
#pragma unroll
                for (int al = 0; al < 3; ++al)
#pragma unroll
                    for (int be = 0; be < 3; ++be) cmac(e[al], D[3 * al + be], g.mom[3 * d + be]);
            }
        }
#pragma unroll
        for (int al = 0; al < 3; ++al) B[t * m + 3 * l + al] = e[al];
    }
    __syncthreads();
    {   // C_f = A^+ B_f: a thread makes one unknown of half the functions
        constexpr int half = kFunPerCta / 2;
        const int u = threadIdx.x % kNU, t0 = threadIdx.x / kNU * half;
        double2 acc[half];
#pragma unroll
        for (int t = 0; t < half; ++t) acc[t] = make_double2(0.0, 0.0);
#pragma unroll 2
        for (int i = 0; i < m; ++i) {
            const double2 w = g.Apinv[(size_t)i * kNU + u];
#pragma unroll
            for (int t = 0; t < half; ++t) cmac(acc[t], w, B[(t0 + t) * m + i]);
        }
#pragma unroll
        for (int t = 0; t < half; ++t) {
            C[(t0 + t) * kNU + u] = acc[t];
            if (f0 + t0 + t < g.n_fun) g.P[(f0 + t0 + t) * kNU + u] = acc[t];
        }
    }
    if (!g.res) return;
    __syncthreads();
    double rr[kFunPerCta], bb[kFunPerCta];
#pragma unroll
    for (int t = 0; t < kFunPerCta; ++t) rr[t] = bb[t] = 0.0;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double2 s[kFunPerCta];
#pragma unroll
        for (int t = 0; t < kFunPerCta; ++t) s[t] = make_double2(0.0, 0.0);
#pragma unroll 2
        for (int u = 0; u < kNU; ++u) {
            const double2 a = g.A0[i + (size_t)m * u];
#pragma unroll
            for (int t = 0; t < kFunPerCta; ++t) cmac(s[t], a, C[t * kNU + u]);
        }
#pragma unroll
        for (int t = 0; t < kFunPerCta; ++t) {
            const double2 b = B[t * m + i];
            const double dx = s[t].x - b.x, dy = s[t].y - b.y;
            rr[t] += dx * dx + dy * dy;
            bb[t] += b.x * b.x + b.y * b.y;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int t = 0; t < kFunPerCta; ++t) {
        for (int o = 16; o; o >>= 1) {
            rr[t] += __shfl_xor_sync(0xffffffffu, rr[t], o);
            bb[t] += __shfl_xor_sync(0xffffffffu, bb[t], o);
        }
        if (lane == 0) {
            red[0][t][warp] = rr[t];
            red[1][t][warp] = bb[t];
        }
    }
    __syncthreads();
    if (threadIdx.x < kFunPerCta) {
        const int t = threadIdx.x;
        double r2 = 0.0, b2 = 0.0;
        for (int w = 0; w < kMapThreads / 32; ++w) {
            r2 += red[0][t][w];
            b2 += red[1][t][w];
        }
        if (f0 + t < g.n_fun) g.res[f0 + t] = b2 > 0.0 ? sqrt(r2 / b2) : 0.0;
    }
}

// Device buffers of one ie_map_basis call, cut from one allocation (an allocation and its
// release take about 0.1 ms each), freed on every return path.
struct Scratch {
    char *base = nullptr;
    size_t used = 0;
    ~Scratch() {
        if (base) cudaFree(base);
    }
    static size_t round(size_t bytes) { return (bytes + 255) / 256 * 256; }
    ie_status reserve(size_t bytes) {
        cudaError_t e = cudaMalloc((void **)&base, bytes);
        if (e == cudaSuccess) return IE_OK;
        base = nullptr;
        cudaGetLastError();
        set_error("cudaMalloc(%zu bytes): %s", bytes, cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? IE_ERR_OOM : IE_ERR_CUDA;
    }
    template <class T>
    T *get(size_t count) {
        T *p = reinterpret_cast<T *>(base + used);
        used += round(count * sizeof(T));
        return p;
    }
};

bool finite_positive(double x) { return std::isfinite(x) && x > 0.0; }

ie_status validate(const ie_mapping_spec *spec, int64_t n_fun, const int64_t *fun_off, const double *pos,
                   const double *mom, const double *P) {
    if (!spec) return set_error("null spec"), IE_ERR_INVALID;
    if (!finite_positive(spec->k) || !finite_positive(spec->eta) || !finite_positive(spec->box_edge))
        return set_error("k, eta and box_edge must be positive and finite"), IE_ERR_INVALID;
    if (spec->lattice != kLattice) return set_error("lattice %d: only 4 is supported", spec->lattice), IE_ERR_INVALID;
    if (spec->n_samples < kMinSamples || spec->n_samples > kMaxSamples)
        return set_error("n_samples %d outside [%d, %d]", spec->n_samples, kMinSamples, kMaxSamples), IE_ERR_INVALID;
    if (!std::isfinite(spec->sample_radius) || !(spec->sample_radius > 0.5 * std::sqrt(3.0)))
        return set_error("sample_radius %g must exceed sqrt(3)/2 (S must enclose the box)", spec->sample_radius),
               IE_ERR_INVALID;
    if (!std::isfinite(spec->tikhonov) || spec->tikhonov < 0.0)
        return set_error("tikhonov %g must be finite and >= 0", spec->tikhonov), IE_ERR_INVALID;
    if (n_fun < 0) return set_error("n_fun %lld < 0", (long long)n_fun), IE_ERR_INVALID;
    if (n_fun == 0) return IE_OK;
    if (!fun_off || !P) return set_error("null fun_off or P"), IE_ERR_INVALID;
    if (fun_off[0] != 0) return set_error("fun_off[0] = %lld, must be 0", (long long)fun_off[0]), IE_ERR_INVALID;
    for (int64_t f = 0; f < n_fun; ++f)
        if (fun_off[f + 1] < fun_off[f])
            return set_error("fun_off decreases at function %lld", (long long)f), IE_ERR_INVALID;
    const int64_t nd = fun_off[n_fun];
    if (nd > 0 && (!pos || !mom)) return set_error("null pos or mom"), IE_ERR_INVALID;
    const double rs = spec->sample_radius * spec->box_edge;
    for (int64_t d = 0; d < nd; ++d) {
        const double *x = pos + 3 * d;
        for (int c = 0; c < 3; ++c)
            if (!std::isfinite(x[c])) return set_error("non-finite position of dipole %lld", (long long)d), IE_ERR_INVALID;
        for (int c = 0; c < 6; ++c)
            if (!std::isfinite(mom[6 * d + c]))
                return set_error("non-finite moment of dipole %lld", (long long)d), IE_ERR_INVALID;
        if (!(std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]) < rs))
            return set_error("dipole %lld lies outside the sampling sphere (radius %g)", (long long)d, rs),
                   IE_ERR_INVALID;
    }
    return IE_OK;
}

}  // namespace
}  // namespace ie

using namespace ie;

extern "C" ie_status ie_map_basis(const ie_mapping_spec *spec, int64_t n_fun, const int64_t *fun_off,
                                  const double *pos, const double *mom, double *P, double *residual,
                                  void *stream) {
    IE_TRY(validate(spec, n_fun, fun_off, pos, mom, P));
    if (n_fun == 0) return IE_OK;
    NvtxRange nv("ie_map_basis");
    cudaStream_t st = (cudaStream_t)stream;
    const Sphere s{spec->k, spec->eta, spec->box_edge, spec->sample_radius * spec->box_edge, spec->n_samples};
    const int m = 3 * s.ns;                                      // rows of A
    const int mf = spec->tikhonov > 0.0 ? m + kNU : m;           // rows of the factorised matrix
    const int64_t chunk = n_fun < kMapChunk ? n_fun : kMapChunk;
    int64_t max_dip = 0;
    for (int64_t f0 = 0; f0 < n_fun; f0 += chunk) {
        int64_t f1 = f0 + chunk < n_fun ? f0 + chunk : n_fun;
        max_dip = std::max(max_dip, fun_off[f1] - fun_off[f0]);
    }
    Scratch sc;
    {
        size_t b = 2 * Scratch::round((size_t)mf * kNU * sizeof(double2)) +
                   2 * Scratch::round((size_t)m * kNU * sizeof(double2)) + Scratch::round(kNU * sizeof(double)) +
                   Scratch::round((kNU + 1) * sizeof(int)) + Scratch::round(((size_t)chunk + 1) * sizeof(int64_t)) +
                   Scratch::round(3 * (size_t)max_dip * sizeof(double)) +
                   Scratch::round(3 * (size_t)max_dip * sizeof(double2)) +
                   Scratch::round((size_t)chunk * kNU * sizeof(double2));
        if (residual) b += Scratch::round((size_t)chunk * sizeof(double));
        IE_TRY(sc.reserve(b));
    }
    double2 *A = sc.get<double2>((size_t)mf * kNU), *V = sc.get<double2>((size_t)mf * kNU);
    double2 *A0 = sc.get<double2>((size_t)m * kNU), *Apinv = sc.get<double2>((size_t)m * kNU);
    double *tau = sc.get<double>(kNU);
    int *flag = sc.get<int>(kNU + 1);
    int64_t *d_off = sc.get<int64_t>((size_t)chunk + 1);
    double *d_pos = sc.get<double>(3 * (size_t)max_dip);
    double2 *d_mom = sc.get<double2>(3 * (size_t)max_dip);
    double2 *d_P = sc.get<double2>((size_t)chunk * kNU);
    double *d_res = residual ? sc.get<double>((size_t)chunk) : nullptr;
    int *status = flag + kNU;
    IE_CK(cudaMemsetAsync(flag, 0, (kNU + 1) * sizeof(int), st));

    sample_matrix_kernel<<<(s.ns * kSites + 255) / 256, 256, 0, st>>>(s, A, mf, A0);
    IE_CK_LAUNCH();
    {   // its CTAs wait on one another: all of them resident
        int mq = mf, md = m;
        double tk = spec->tikhonov;
        void *args[] = {&A, &A0, &mq, &md, &tk, &V, &tau, &flag, &Apinv, &status};
        IE_CK(cudaLaunchCooperativeKernel((const void *)qr_kernel, dim3(kNU), dim3(kQrThreads), args, 0, st));
        IE_CK_LAUNCH();
    }
    int h_status = 0;
    IE_CK(cudaMemcpyAsync(&h_status, status, sizeof(int), cudaMemcpyDeviceToHost, st));
    IE_CK(cudaStreamSynchronize(st));
    if (h_status == 1) return set_error("the uniform-dipole field matrix A is rank deficient"), IE_ERR_INVALID;
    if (h_status) return set_error("the factorisation gave up a bounded wait"), IE_ERR_TIMEOUT;
    pinv_solve_kernel<<<m, 32, 0, st>>>(A, mf, Apinv);
    IE_CK_LAUNCH();

    const size_t map_smem = (size_t)kFunPerCta * (m + kNU) * sizeof(double2);
    IE_CK(cudaFuncSetAttribute(map_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)map_smem));
    std::vector<int64_t> off(chunk + 1);
    for (int64_t f0 = 0; f0 < n_fun; f0 += chunk) {
        const int64_t nf = std::min(chunk, n_fun - f0);
        const int64_t d0 = fun_off[f0], nd = fun_off[f0 + nf] - d0;
        for (int64_t f = 0; f <= nf; ++f) off[f] = fun_off[f0 + f] - d0;
        IE_CK(cudaMemcpyAsync(d_off, off.data(), (nf + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, st));
        if (nd > 0) {
            IE_CK(cudaMemcpyAsync(d_pos, pos + 3 * d0, 3 * nd * sizeof(double), cudaMemcpyHostToDevice, st));
            IE_CK(cudaMemcpyAsync(d_mom, mom + 6 * d0, 3 * nd * sizeof(double2), cudaMemcpyHostToDevice, st));
        }
        MapArgs g{s, nf, d_off, d_pos, d_mom, Apinv, A0, d_P, d_res};
        map_kernel<<<(unsigned)((nf + kFunPerCta - 1) / kFunPerCta), kMapThreads, map_smem, st>>>(g);
        IE_CK_LAUNCH();
        IE_CK(cudaMemcpyAsync(P + 2 * (size_t)f0 * kNU, d_P, (size_t)nf * kNU * sizeof(double2),
                              cudaMemcpyDeviceToHost, st));
        if (residual)
            IE_CK(cudaMemcpyAsync(residual + f0, d_res, nf * sizeof(double), cudaMemcpyDeviceToHost, st));
        // the staging buffers are reused by the next chunk
        IE_CK(cudaStreamSynchronize(st));
    }
    return IE_OK;
}

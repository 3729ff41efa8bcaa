// K3 (lattice form): the far product as a discrete convolution.
//
// The dipoles of all boxes lie on one lattice of spacing h = a / 4, and D (eq. 5) depends on
// the separation only, so with K'(m) = D(h m) for |m|_inf >= 5 and 0 otherwise,
//     (K' * x)(t) = sum over far boxes  +  sum over adjacent boxes of the site pairs with
//                   5 <= |m|_inf <= 7
// (far sites are at least 5 lattice steps apart, sites of adjacent boxes at most 7).  The
// second sum is a product with 26 masked blocks: IE_FULL leaves it inside the convolution
// and applies near blocks cut to |m|_inf <= 4 (no extra work), IE_FAR and ie_translate take
// it off with the block-product kernels over the adjacent pairs (translate_simt.cu,
// translate_tc.cu).  Nothing is added that cancels: all kept and removed terms have the
// size of far interactions, as long as the sources are even enough (kFarEven); inputs that are
// not take the block products.
//
// The convolution runs per scatterer and right-hand side over the scatterer's bounding
// lattice (n_i = 4 E_i sites per axis, zero-padded to L_i >= 2 n_i - 1) in five passes:
//     x lines of the boxes' sites -> A[c][z][y][kx]       (n_z n_y lines of L_x)
//     y: A -> B[c][z][ky][kx]                             (only the n_y occupied rows read)
//     z: per (ky, kx) the three components together: transform, multiply with the 3 x 3
//        symmetric tensor K^, transform back, B in place  (only n_z planes read and written)
//     y back: B -> A,  x back: A -> the boxes' sites.
// So the padded cube itself is never stored: the z pass holds its lines in shared memory.
// K^ comes from FP64 sums (separable cosine / sine sums over the octant, K' being even or
// odd along each axis), rounded once to FP32, with 1 / (L_x L_y L_z) folded in.
//
// Cost: O(L^3 log L) instead of 192^2 multiply-adds per far pair.  Measured far part of one
// IE_FULL product: 0.39 ms on the 32^3 shell (L = 256: x 26, y 52, z 231, y back 49, x back
// 28 us) against 17.7 ms (FP16X3) and 150 ms (FP32) of the block products; 0.064 ms on the
// 16^3 shell (L = 128) against 1.5 and 12.2 ms.
#include <algorithm>
#include <array>
#include <climits>
#include <cmath>
#include <utility>

#include "ie_internal.h"

namespace ie {
namespace {

// ---------------------------------------------------------------- small transforms in registers
constexpr double kPi = 3.14159265358979323846;
// Taylor series after reduction to [-pi/4, pi/4]: compile-time constants only
constexpr double sin_small(double x) {
    double t = x, s = x;
    for (int i = 1; i < 12; ++i) t *= -x * x / ((2 * i) * (2 * i + 1)), s += t;
    return s;
}
constexpr double cos_small(double x) {
    double t = 1, s = 1;
    for (int i = 1; i < 12; ++i) t *= -x * x / ((2 * i - 1) * (2 * i)), s += t;
    return s;
}
// cos / sin of 2 pi k / n
constexpr double cos_turn(int k, int n) {
    k = ((k % n) + n) % n;
    if (2 * k > n) k = n - k;
    if (4 * k > n) return -cos_turn(n - 2 * k, 2 * n);
    if (8 * k > n) return sin_small(2 * kPi * (n - 4 * k) / (4.0 * n));
    return cos_small(2 * kPi * k / n);
}
constexpr double sin_turn(int k, int n) { return cos_turn(4 * k - n, 4 * n); }

template <class F, int... I>
__device__ __forceinline__ void unroll_impl(F &&f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void unroll(F &&f) {
    unroll_impl(f, std::make_integer_sequence<int, N>{});
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmulf(float2 a, float2 w) {
    return make_float2(fmaf(a.x, w.x, -a.y * w.y), fmaf(a.x, w.y, a.y * w.x));
}
// a * exp(DIR 2 pi i K / N)
template <int K, int N, int DIR>
__device__ __forceinline__ float2 twiddle(float2 a) {
    constexpr int k = ((K % N) + N) % N;
    if constexpr (k == 0) {
        return a;
    } else if constexpr (4 * k == N) {
        return DIR > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
    } else if constexpr (2 * k == N) {
        return make_float2(-a.x, -a.y);
    } else if constexpr (4 * k == 3 * N) {
        return DIR > 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
    } else {
        constexpr float c = (float)cos_turn(k, N), s = (float)(DIR * sin_turn(k, N));
        return cmulf(a, make_float2(c, s));
    }
}

template <int R, int DIR>
__device__ __forceinline__ void dft(float2 (&v)[R]);

template <int A, int B, int DIR>
__device__ __forceinline__ void dft_split(float2 (&v)[A * B]) {
    float2 t[B][A];
    unroll<B>([&](auto b) {
        float2 u[A];
        unroll<A>([&](auto a) { u[a] = v[B * a + b]; });
        dft<A, DIR>(u);
        unroll<A>([&](auto k) {
            constexpr int e = decltype(b)::value * decltype(k)::value;
            t[b][k] = twiddle<e, A * B, DIR>(u[k]);
        });
    });
    unroll<A>([&](auto k1) {
        float2 u[B];
        unroll<B>([&](auto b) { u[b] = t[b][k1]; });
        dft<B, DIR>(u);
        unroll<B>([&](auto k2) { v[k1 + A * k2] = u[k2]; });
    });
}

// v[k] <- sum_n v[n] exp(DIR 2 pi i n k / R)
template <int R, int DIR>
__device__ __forceinline__ void dft(float2 (&v)[R]) {
    if constexpr (R == 2) {
        const float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (R == 3) {
        constexpr float s = (float)(DIR * sin_turn(1, 3));
        const float2 t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
        const float2 m = make_float2(fmaf(-0.5f, t.x, v[0].x), fmaf(-0.5f, t.y, v[0].y));
        v[0] = cadd(v[0], t);
        v[1] = make_float2(fmaf(-s, d.y, m.x), fmaf(s, d.x, m.y));
        v[2] = make_float2(fmaf(s, d.y, m.x), fmaf(-s, d.x, m.y));
    } else if constexpr (R == 4) {
        const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
        const float2 e = DIR > 0 ? make_float2(-d.y, d.x) : make_float2(d.y, -d.x);
        v[0] = cadd(a, c);
        v[1] = cadd(b, e);
        v[2] = csub(a, c);
        v[3] = csub(b, e);
    } else if constexpr (R % 4 == 0) {
        dft_split<4, R / 4, DIR>(v);
    } else {
        static_assert(R % 2 == 0, "radices 2^a 3^b");
        dft_split<2, R / 2, DIR>(v);
    }
}

// Forward transform of R values whose upper half is zero (v[0 .. R/2) given).
template <int R>
__device__ __forceinline__ void dft_half_in(float2 (&v)[R]) {
    constexpr int H = R / 2;
    float2 e[H], o[H];
    unroll<H>([&](auto a) {
        e[a] = v[a];
        o[a] = twiddle<decltype(a)::value, R, -1>(v[a]);
    });
    dft<H, -1>(e);
    dft<H, -1>(o);
    unroll<H>([&](auto j) {
        v[2 * j] = e[j];
        v[2 * j + 1] = o[j];
    });
}
// Backward transform of R values, the lower half of the result only (v[0 .. R/2)).
template <int R>
__device__ __forceinline__ void dft_half_out(float2 (&v)[R]) {
    constexpr int H = R / 2;
    float2 e[H], o[H];
    unroll<H>([&](auto j) {
        e[j] = v[2 * j];
        o[j] = v[2 * j + 1];
    });
    dft<H, 1>(e);
    dft<H, 1>(o);
    unroll<H>([&](auto a) { v[a] = cadd(e[a], twiddle<decltype(a)::value, R, 1>(o[a])); });
}

// ---------------------------------------------------------------- passes
// A line of L = R1 R2 points: n = R2 a + b, k = k1 + R1 k2,
//   X[k1 + R1 k2] = sum_b w_R2^(b k2) w_L^(b k1) sum_a w_R1^(a k1) x[R2 a + b].
// Forward: the a sums (upper half of a is padding), one exchange through shared memory, the
// b sums.  Backward in the opposite order, so no pass reorders anything.
struct ConvArgs {
    const float2 *X;            // [rhs][nbox][192]
    float2 *Y;                  // [rhs][nbox][192]
    float2 *A, *B;              // per column a_col / b_col elements
    int64_t a_col, b_col;
    const float4 *K;            // [xx xy | xz yy | yz zz][kz][ky][kx], octant
    const int32_t *slot;        // [scatterer][Ez][Ey][Ex] box, or -1
    const int32_t *cols;        // [scatterer] right-hand sides it takes part with
    const float2 *twx, *twy, *twz;   // exp(-2 pi i j / L)
    int Ex, Ey, Ez, Lx, Ly, Lz;
    int nbox, nrhs, q0;         // column q0 + blockIdx.z: scatterer q / nrhs, right-hand side q % nrhs
    const int *gate;
};

constexpr int kW = 16;              // lines per tile of the y and z passes: 128-byte rows
// x lines per CTA: rows of sites so that each first-stage thread has one sum to do
template <int R2>
struct XTile {
    static constexpr int rows = 64 / R2;          // 3 rows R2 = 192 sums
};
constexpr int kXThreads = 192;

// shared memory of one x line: [k1][b], rows padded to an odd length, lines skewed
template <int R1, int R2>
constexpr int x_line() { return R1 * (R2 + 1) + 5; }

template <int R1, int R2>
__global__ void __launch_bounds__(kXThreads) conv_x_kernel(const ConvArgs a) {
    chain_wait();
    if (a.gate && *a.gate == 0) return;
    constexpr int L = R1 * R2, rows = XTile<R2>::rows, LS = x_line<R1, R2>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *S = reinterpret_cast<float2 *>(smem_raw);
    float2 *tw = S + 3 * rows * LS;
    const int q = a.q0 + blockIdx.z, s = q / a.nrhs, r = q - s * a.nrhs;
    if (r >= a.cols[s]) return;
    const int y0 = blockIdx.x * rows, z = blockIdx.y, ny = 4 * a.Ey, nx = 4 * a.Ex;
    for (int i = threadIdx.x; i < L; i += kXThreads) tw[i] = a.twx[i];
    __syncthreads();
    {
        const int c = threadIdx.x % 3, b = (threadIdx.x / 3) % R2, row = threadIdx.x / (3 * R2), y = y0 + row;
        float2 v[R1];
        const int32_t *sl = a.slot + (((int64_t)s * a.Ez + (z >> 2)) * a.Ey + (y >> 2)) * a.Ex;
        const float2 *x = a.X + (int64_t)r * a.nbox * kNU + 12 * (y & 3) + 48 * (z & 3) + c;
        unroll<R1 / 2>([&](auto i) {
            const int n = R2 * i + b;
            v[i] = make_float2(0.f, 0.f);
            if (y < ny && n < nx) {
                const int box = __ldg(sl + (n >> 2));
                if (box >= 0) v[i] = x[(int64_t)box * kNU + 3 * (n & 3)];
            }
        });
        dft_half_in<R1>(v);
        float2 *d = S + (row * 3 + c) * LS + b;
        unroll<R1>([&](auto k) { d[k * (R2 + 1)] = cmulf(v[k], tw[b * k]); });
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 3 * rows * R1; t += kXThreads) {
        const int k1 = t % R1, line = t / R1, c = line % 3, y = y0 + line / 3;
        if (y >= ny) continue;
        float2 v[R2];
        const float2 *d = S + line * LS + k1 * (R2 + 1);
        unroll<R2>([&](auto b) { v[b] = d[b]; });
        dft<R2, -1>(v);
        float2 *out = a.A + blockIdx.z * a.a_col + (((int64_t)c * (4 * a.Ez) + z) * ny + y) * L + k1;
        unroll<R2>([&](auto k2) { out[R1 * k2] = v[k2]; });
    }
}

template <int R1, int R2>
__global__ void __launch_bounds__(kXThreads) conv_xback_kernel(const ConvArgs a) {
    chain_wait();
    if (a.gate && *a.gate == 0) return;
    constexpr int L = R1 * R2, rows = XTile<R2>::rows, LS = x_line<R1, R2>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *S = reinterpret_cast<float2 *>(smem_raw);
    float2 *tw = S + 3 * rows * LS;
    const int q = a.q0 + blockIdx.z, s = q / a.nrhs, r = q - s * a.nrhs;
    const bool on = r < a.cols[s];      // a column the scatterer does not have: zero field
    const int y0 = blockIdx.x * rows, z = blockIdx.y, ny = 4 * a.Ey, nx = 4 * a.Ex;
    if (on) {
        for (int i = threadIdx.x; i < L; i += kXThreads) tw[i] = a.twx[i];
        __syncthreads();
        for (int t = threadIdx.x; t < 3 * rows * R1; t += kXThreads) {
            const int k1 = t % R1, line = t / R1, c = line % 3, y = y0 + line / 3;
            if (y >= ny) continue;
            float2 v[R2];
            const float2 *in = a.A + blockIdx.z * a.a_col + (((int64_t)c * (4 * a.Ez) + z) * ny + y) * L + k1;
            unroll<R2>([&](auto k2) { v[k2] = in[R1 * k2]; });
            dft<R2, 1>(v);
            float2 *d = S + line * LS + k1 * (R2 + 1);
            unroll<R2>([&](auto b) {
                const float2 w = tw[b * k1];
                d[b] = cmulf(v[b], make_float2(w.x, -w.y));
            });
        }
        __syncthreads();
    }
    const int c = threadIdx.x % 3, b = (threadIdx.x / 3) % R2, row = threadIdx.x / (3 * R2), y = y0 + row;
    if (y >= ny) return;
    float2 v[R1];
    if (on) {
        const float2 *d = S + (row * 3 + c) * LS + b;
        unroll<R1>([&](auto k) { v[k] = d[k * (R2 + 1)]; });
        dft_half_out<R1>(v);
    } else {
        unroll<R1>([&](auto k) { v[k] = make_float2(0.f, 0.f); });
    }
    const int32_t *sl = a.slot + (((int64_t)s * a.Ez + (z >> 2)) * a.Ey + (y >> 2)) * a.Ex;
    float2 *out = a.Y + (int64_t)r * a.nbox * kNU + 12 * (y & 3) + 48 * (z & 3) + c;
    unroll<R1 / 2>([&](auto i) {
        const int n = R2 * i + b;
        if (n < nx) {
            const int box = __ldg(sl + (n >> 2));
            if (box >= 0) out[(int64_t)box * kNU + 3 * (n & 3)] = v[i];
        }
    });
}

// y pass of one (component, plane z, kx tile)
template <int R1, int R2>
__global__ void __launch_bounds__(kW *R2) conv_y_kernel(const ConvArgs a) {
    chain_wait();
    if (a.gate && *a.gate == 0) return;
    constexpr int L = R1 * R2, NT = kW * R2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *S = reinterpret_cast<float2 *>(smem_raw);           // [L][kW]
    float2 *tw = S + L * kW;
    const int q = a.q0 + blockIdx.z / 3, s = q / a.nrhs, c = blockIdx.z % 3;
    if (q - s * a.nrhs >= a.cols[s]) return;
    const int z = blockIdx.y, ny = 4 * a.Ey, nz = 4 * a.Ez, w = threadIdx.x % kW;
    const float2 *in = a.A + (blockIdx.z / 3) * a.a_col + ((int64_t)c * nz + z) * ny * a.Lx + blockIdx.x * kW + w;
    float2 *out = a.B + (blockIdx.z / 3) * a.b_col + ((int64_t)c * nz + z) * L * a.Lx + blockIdx.x * kW + w;
    for (int i = threadIdx.x; i < L; i += NT) tw[i] = a.twy[i];
    {
        const int b = threadIdx.x / kW;
        float2 v[R1];
        unroll<R1 / 2>([&](auto i) {
            const int y = R2 * i + b;
            v[i] = y < ny ? in[(int64_t)y * a.Lx] : make_float2(0.f, 0.f);
        });
        dft_half_in<R1>(v);
        __syncthreads();
        unroll<R1>([&](auto k) { S[(k * R2 + b) * kW + w] = cmulf(v[k], tw[b * k]); });
    }
    __syncthreads();
    for (int k1 = threadIdx.x / kW; k1 < R1; k1 += R2) {
        float2 v[R2];
        unroll<R2>([&](auto b) { v[b] = S[(k1 * R2 + b) * kW + w]; });
        dft<R2, -1>(v);
        unroll<R2>([&](auto k2) { out[(int64_t)(k1 + R1 * k2) * a.Lx] = v[k2]; });
    }
}

template <int R1, int R2>
__global__ void __launch_bounds__(kW *R2) conv_yback_kernel(const ConvArgs a) {
    chain_wait();
    if (a.gate && *a.gate == 0) return;
    constexpr int L = R1 * R2, NT = kW * R2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *S = reinterpret_cast<float2 *>(smem_raw);           // [L][kW]
    float2 *tw = S + L * kW;
    const int q = a.q0 + blockIdx.z / 3, s = q / a.nrhs, c = blockIdx.z % 3;
    if (q - s * a.nrhs >= a.cols[s]) return;
    const int z = blockIdx.y, ny = 4 * a.Ey, nz = 4 * a.Ez, w = threadIdx.x % kW;
    float2 *out = a.A + (blockIdx.z / 3) * a.a_col + ((int64_t)c * nz + z) * ny * a.Lx + blockIdx.x * kW + w;
    const float2 *in = a.B + (blockIdx.z / 3) * a.b_col + ((int64_t)c * nz + z) * L * a.Lx + blockIdx.x * kW + w;
    for (int i = threadIdx.x; i < L; i += NT) tw[i] = a.twy[i];
    __syncthreads();
    for (int k1 = threadIdx.x / kW; k1 < R1; k1 += R2) {
        float2 v[R2];
        unroll<R2>([&](auto k2) { v[k2] = in[(int64_t)(k1 + R1 * k2) * a.Lx]; });
        dft<R2, 1>(v);
        unroll<R2>([&](auto b) {
            const float2 t = tw[b * k1];
            S[(k1 * R2 + b) * kW + w] = cmulf(v[b], make_float2(t.x, -t.y));
        });
    }
    __syncthreads();
    const int b = threadIdx.x / kW;
    float2 v[R1];
    unroll<R1>([&](auto k) { v[k] = S[(k * R2 + b) * kW + w]; });
    dft_half_out<R1>(v);
    unroll<R1 / 2>([&](auto i) {
        const int y = R2 * i + b;
        if (y < ny) out[(int64_t)y * a.Lx] = v[i];
    });
}

__device__ __forceinline__ void cmac(float2 &d, float2 a, float2 b) {
    d.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, d.x));
    d.y = fmaf(a.x, b.y, fmaf(a.y, b.x, d.y));
}

// z pass of one (ky, kx tile): transform, tensor product, transform back, in place.  Blocks
// of mirrored (ky, kx) run next to each other, so that the octant of K^ they share is read
// from device memory once.
//
// Bound by latency (loads of K^ and of the lines) at the occupancy that shared memory (24 L kW
// bytes) and registers (three components of an R2-point sum) leave: 46% of the issue slots at L
// = 256 with two CTAs per SM, 231 us on the 32^3 shell; one CTA per SM and K^ as 48-byte records
// took 340 us.  Up to L = 192 the registers hold K^ points and lines ahead (16^3 shell 32 -> 29
// us, 4^3 grid 9.8 -> 6.4); at L = 256 they do not (lines ahead 318 us, R1 = 32 with K^ ahead but
// half the threads 254, tiles of 8 lines 253).
// PFMAX: points of K^ fetched ahead of their use; AHEAD: the three components' lines too.
template <int R1, int R2, int PFMAX, bool AHEAD, int CTAS>
__global__ void __launch_bounds__(kW *R2, CTAS) conv_z_kernel(const ConvArgs a) {
    chain_wait();
    if (a.gate && *a.gate == 0) return;
    constexpr int L = R1 * R2, NT = kW * R2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *S = reinterpret_cast<float2 *>(smem_raw);           // [3][L][kW]
    float2 *tw = S + 3 * L * kW;
    const int q = a.q0 + blockIdx.z, s = q / a.nrhs;
    if (q - s * a.nrhs >= a.cols[s]) return;
    const int w = threadIdx.x % kW, b0 = threadIdx.x / kW, nz = 4 * a.Ez;
    const int xt = (blockIdx.x & 1) ? gridDim.x - 1 - (blockIdx.x >> 1) : (blockIdx.x >> 1);
    const int kx = xt * kW + w;
    const int ky = (blockIdx.y & 1) ? a.Ly - 1 - (blockIdx.y >> 1) : (blockIdx.y >> 1);
    const int64_t plane = (int64_t)a.Ly * a.Lx;
    float2 *B = a.B + blockIdx.z * a.b_col + (int64_t)ky * a.Lx + kx;
    auto load = [&](int c, float2(&u)[R1 / 2]) {
        unroll<R1 / 2>([&](auto i) {
            const int z = R2 * i + b0;
            u[i] = z < nz ? B[(int64_t)(c * nz + z) * plane] : make_float2(0.f, 0.f);
        });
    };
    auto first = [&](int c, const float2(&u)[R1 / 2]) {
        float2 v[R1];
        unroll<R1 / 2>([&](auto i) { v[i] = u[i]; });
        dft_half_in<R1>(v);
        unroll<R1>([&](auto k) { S[((c * R1 + k) * R2 + b0) * kW + w] = cmulf(v[k], tw[b0 * k]); });
    };
    if constexpr (AHEAD) {      // all three components' loads in flight together
        float2 u[3][R1 / 2];
        unroll<3>([&](auto c) { load(c, u[c]); });
        for (int i = threadIdx.x; i < L; i += NT) tw[i] = a.twz[i];
        __syncthreads();
        unroll<3>([&](auto c) { first(c, u[c]); });
    } else {
        for (int i = threadIdx.x; i < L; i += NT) tw[i] = a.twz[i];
        __syncthreads();
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
            float2 u[R1 / 2];
            load(c, u);
            first(c, u);
        }
    }
    __syncthreads();
    const int ax = 2 * kx > a.Lx ? a.Lx - kx : kx, ay = 2 * ky > a.Ly ? a.Ly - ky : ky;
    const float sx = 2 * kx > a.Lx ? -1.f : 1.f, sy = 2 * ky > a.Ly ? -1.f : 1.f;
    const int mx = a.Lx / 2 + 1, my = a.Ly / 2 + 1;
    const int64_t kpart = (int64_t)(L / 2 + 1) * my * mx;
    constexpr int PF = R2 < PFMAX ? R2 : PFMAX;
    for (int k1 = b0; k1 < R1; k1 += R2) {
        float4 f[PF][3];
        auto fetch = [&](int k2, float4(&g)[3]) {
            const int kz = k1 + R1 * k2;
            const int az = 2 * kz > L ? L - kz : kz;
            const float4 *K = a.K + ((int64_t)az * my + ay) * mx + ax;
            g[0] = __ldg(K), g[1] = __ldg(K + kpart), g[2] = __ldg(K + 2 * kpart);
        };
        unroll<PF>([&](auto i) { fetch(i, f[i]); });
        float2 v[3][R2];
        unroll<3>([&](auto c) {
            unroll<R2>([&](auto b) { v[c][b] = S[((c * R1 + k1) * R2 + b) * kW + w]; });
            dft<R2, -1>(v[c]);
        });
        unroll<R2>([&](auto k2) {
            constexpr int at = decltype(k2)::value % PF;
            const float sz = 2 * (k1 + R1 * k2) > L ? -1.f : 1.f;
            const float4 f0 = f[at][0], f1 = f[at][1], f2 = f[at][2];
            if constexpr (decltype(k2)::value + PF < R2) fetch(k2 + PF, f[at]);
            const float sxy = sx * sy, sxz = sx * sz, syz = sy * sz;
            const float2 xx = make_float2(f0.x, f0.y), xy = make_float2(sxy * f0.z, sxy * f0.w);
            const float2 xz = make_float2(sxz * f1.x, sxz * f1.y), yy = make_float2(f1.z, f1.w);
            const float2 yz = make_float2(syz * f2.x, syz * f2.y), zz = make_float2(f2.z, f2.w);
            const float2 x = v[0][k2], y = v[1][k2], z = v[2][k2];
            float2 o0 = make_float2(0.f, 0.f), o1 = o0, o2 = o0;
            cmac(o0, xx, x), cmac(o0, xy, y), cmac(o0, xz, z);
            cmac(o1, xy, x), cmac(o1, yy, y), cmac(o1, yz, z);
            cmac(o2, xz, x), cmac(o2, yz, y), cmac(o2, zz, z);
            v[0][k2] = o0, v[1][k2] = o1, v[2][k2] = o2;
        });
        unroll<3>([&](auto c) {
            dft<R2, 1>(v[c]);
            unroll<R2>([&](auto b) {
                const float2 t = tw[b * k1];
                S[((c * R1 + k1) * R2 + b) * kW + w] = cmulf(v[c][b], make_float2(t.x, -t.y));
            });
        });
    }
    __syncthreads();
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
        float2 v[R1];
        unroll<R1>([&](auto k) { v[k] = S[((c * R1 + k) * R2 + b0) * kW + w]; });
        dft_half_out<R1>(v);
        unroll<R1 / 2>([&](auto i) {
            const int z = R2 * i + b0;
            if (z < nz) B[((int64_t)c * nz + z) * plane] = v[i];
        });
    }
}

// The supported line lengths and their two factors (R1 even; R1, R2 of the form 2^a 3^b).
#define IE_CONV_SIZES(F) \
    F(16, 4, 4) F(32, 8, 4) F(48, 12, 4) F(64, 8, 8) F(96, 12, 8) F(128, 16, 8) F(192, 24, 8) F(256, 16, 16) \
    F(384, 24, 16) F(512, 32, 16)
// z lines: K^ points ahead, lines ahead, CTAs per SM (shared memory and registers)
#define IE_CONV_ZSIZES(F)                                                                                    \
    F(16, 4, 4, 4, true, 8) F(32, 8, 4, 4, true, 8) F(48, 12, 4, 4, true, 8) F(64, 8, 8, 4, true, 4)         \
    F(96, 12, 8, 4, true, 4) F(128, 16, 8, 4, true, 4) F(192, 24, 8, 4, false, 3) F(256, 16, 16, 1, false, 2) \
    F(384, 24, 16, 2, false, 1) F(512, 32, 16, 2, false, 1)

template <int R1, int R2>
constexpr size_t x_smem() { return (size_t)(3 * XTile<R2>::rows * x_line<R1, R2>() + R1 * R2) * sizeof(float2); }
template <int R1, int R2>
constexpr size_t y_smem() { return (size_t)(R1 * R2 * kW + R1 * R2) * sizeof(float2); }
template <int R1, int R2>
constexpr size_t z_smem() { return (size_t)(3 * R1 * R2 * kW + R1 * R2) * sizeof(float2); }

// ---------------------------------------------------------------- K^ (plan creation)
// One component of K' on the octant, FP64: T[mz][my][mx], 0 <= m_i < n_i.
__global__ void conv_green_kernel(double k, double eta, double h, int nx, int ny, int nz, int i, int j,
                                  double2 *__restrict__ T) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)nx * ny * nz) return;
    const int mx = (int)(t % nx), my = (int)((t / nx) % ny), mz = (int)(t / ((int64_t)nx * ny));
    double2 D[9];
    double2 v = make_double2(0, 0);
    if (max(mx, max(my, mz)) > kNearReach) {
        dyad_fp64(k, eta, h * mx, h * my, h * mz, D);
#pragma unroll
        for (int e = 0; e < 9; ++e)
            if (e == 3 * i + j) v = D[e];
    }
    T[t] = v;
}

// out[o][k][i] = sum_m f(m, k) in[o][m][i], f = cos (weights 1, 2, 2, ..) or 2 sin of
// 2 pi m k / L: the transform of an even or odd sequence along one axis.  A thread makes k
// and L/2 - k from the sums over even and odd m.  FP64 rate bound (7 ms for n = 120, L = 256,
// all three axes and six components).
constexpr int kCt = 16;
__global__ void conv_axis_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, float2 *__restrict__ out32,
                                 double scale, int n, int L, int64_t inner, int64_t cols, int odd,
                                 const double *__restrict__ cs) {
    __shared__ double M[kCt][kCt + 1];
    __shared__ double2 T[kCt][kCt + 1];
    const int K = L / 2 + 1, tx = threadIdx.x % kCt, ty = threadIdx.x / kCt;
    const int k0 = blockIdx.y * kCt, k = k0 + ty;
    const int64_t c0 = (int64_t)blockIdx.x * kCt;
    double2 e = make_double2(0, 0), o = e;
    for (int m0 = 0; m0 < n; m0 += kCt) {
        __syncthreads();
        {   // f(m0 + tx, k0 + ty)
            const int m = m0 + tx, j = (int)((int64_t)m * k % L);
            const double f = odd ? 2 * cs[(j + 3 * L / 4) % L] : (m == 0 ? 1.0 : 2 * cs[j]);
            M[ty][tx] = (m < n && k < K) ? f : 0.0;
        }
        {   // inner = 1: consecutive m are adjacent; otherwise consecutive columns are
            const int mm = inner == 1 ? tx : ty, cc = inner == 1 ? ty : tx;
            const int64_t c = c0 + cc;
            const int m = m0 + mm;
            T[mm][cc] = (m < n && c < cols) ? in[(c / inner) * (n * inner) + m * inner + c % inner] : make_double2(0, 0);
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kCt; m += 2) {
            const double f0 = M[ty][m], f1 = M[ty][m + 1];
            const double2 a = T[m][tx], b = T[m + 1][tx];
            e.x = fma(f0, a.x, e.x), e.y = fma(f0, a.y, e.y);
            o.x = fma(f1, b.x, o.x), o.y = fma(f1, b.y, o.y);
        }
    }
    const int64_t c = c0 + tx;
    if (c >= cols) return;
    auto put = [&](int kk, double re, double im) {
        const int64_t at = (c / inner) * (K * inner) + kk * inner + c % inner;
        if (out32)
            out32[2 * at] = make_float2((float)(scale * re), (float)(scale * im));
        else
            out[at] = make_double2(re, im);
    };
    if (4 * k <= L) put(k, e.x + o.x, e.y + o.y);
    if (4 * k < L) {
        const double g = odd ? -1.0 : 1.0;
        put(L / 2 - k, g * (e.x - o.x), g * (e.y - o.y));
    }
}

int pad_length(int n) {
#define IE_TAKE(L, R1, R2) \
    if (2 * n - 1 <= L) return L;
    IE_CONV_SIZES(IE_TAKE)
#undef IE_TAKE
    return 0;
}

template <int R1, int R2>
ie_status set_attr() {
    IE_CK(cudaFuncSetAttribute(conv_x_kernel<R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x_smem<R1, R2>()));
    IE_CK(cudaFuncSetAttribute(conv_xback_kernel<R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)x_smem<R1, R2>()));
    IE_CK(cudaFuncSetAttribute(conv_y_kernel<R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)y_smem<R1, R2>()));
    IE_CK(cudaFuncSetAttribute(conv_yback_kernel<R1, R2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)y_smem<R1, R2>()));
    return IE_OK;
}

}  // namespace

ie_status prepare_conv() {
#define IE_ATTR(L, R1, R2) IE_TRY((set_attr<R1, R2>()));
    IE_CONV_SIZES(IE_ATTR)
#undef IE_ATTR
#define IE_ATTR(L, R1, R2, PF, AHEAD, CTAS)                                                                         \
    IE_CK(cudaFuncSetAttribute(conv_z_kernel<R1, R2, PF, AHEAD, CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                               (int)z_smem<R1, R2>()));
    IE_CONV_ZSIZES(IE_ATTR)
#undef IE_ATTR
    return IE_OK;
}

// ---------------------------------------------------------------- plan
// Bounds of the rule.  kConvKa: the transforms' rounding is relative to the whole field, so
// the real and imaginary parts of D must be of one size for both to keep FP32 accuracy.  At
// lambda / 8 (k a = 0.785) they are (radiative part of a far product of 6^3 boxes, real moments:
// 2.7e-7, lambda / 4 2.3e-7); at lambda / 256 the radiative part is 1e-4 of the field and a complex
// transform would leave 1e-3 of it.  Nothing between the two is measured: the line lies just
// below lambda / 8.
constexpr double kConvKa = 0.75;
// Device times (ns) of a padded lattice point here, and of a far pair and a stored block (an
// item's chain, however few its pairs) in the block products, 16-bit split and FP32.  They
// place the line for scatterers that are sparse in their bounding box; measured with random
// boxes on grids of 3^3 to 64^3, e.g. 600 boxes on 24^3 249 us here against 441 us (FP16X3),
// 200 boxes 243 against 179; 1,200 boxes on 64^3 4.1 ms against 3.0 ms.
constexpr double kPointNs = 0.03, kPairNs16 = 0.7, kBlockNs16 = 49, kPairNs32 = 6.0, kBlockNs32 = 270;
// A far product alone also takes the adjacent pairs off (a second kernel's chain) and looks at its
// inputs: below this many far pairs the block product is the shorter chain.  Blocks against
// convolution, symmetric store: FP32 5,650 pairs 87 against 105 us without the look, 13,428
// pairs 143 against 103 with it; FP16X3 13,428 pairs 45 against 65 (three columns 78 against 70), 42,560 pairs 70 against 66
// (150 against 70).  One line for all: a single 16-bit column would draw it at 40,000, several at 10,000.
constexpr int64_t kFarPairs = 8192;
constexpr size_t kConvWorkspace = (size_t)256 << 20;    // bytes of A and B beyond one column
// The transforms round relative to the scatterer's whole field, a block product relative to what
// reaches a box, and a far product leaves out what a box's own neighbourhood radiates.  So it is
// a convolution only where, for every box and column, the far boxes hold at least 1 / kFarEven of
// the sources' energy sum |x|^2: the worst box's rounding grows with the square root of that
// ratio (6^3 boxes, one of them A above the rest, FP32: 4e-7 at A = 1, 7e-6 at 1e2, 7e-4 at 1e4;
// blocks 5e-7 throughout).  Inputs that are not so even (a lone source, whose neighbourhood then
// stays exactly zero, strong contrasts, NaN, infinities, or energies so large or small that a
// transform's partial sums could leave FP32's range) take the block products, as decided on the
// device for each call (launch_choose_form).  A plan in which even inputs already fail, because
// some box has less than 1 / kFarEven of its scatterer far from it, keeps the blocks.
constexpr double kFarEven = 4, kEnergyMin = 1e-60, kEnergyMax = 1e60;

ConvUse conv_classes(const ie_problem *pr, int64_t npairs, int64_t nblocks, const std::vector<int32_t> &near_start,
                     std::vector<ConvClass> &out) {
    out.clear();
    unsigned mask = pr->prec_mask & kConvMask;
    if ((int64_t)pr->max_rhs * pr->n_boxes * kNU > (int64_t)INT32_MAX)   // the 16-bit forms' limit
        mask &= IE_PRECMASK(IE_PREC_FP32);
    if (!mask || npairs == 0 || !(pr->k * pr->box_edge >= kConvKa)) return {};
    const int G = pr->box_group ? pr->n_groups : 1;
    std::vector<std::array<int, 6>> bb(G, {INT_MAX, INT_MAX, INT_MAX, INT_MIN, INT_MIN, INT_MIN});
    for (int b = 0; b < pr->n_boxes; ++b) {
        auto &q = bb[pr->box_group ? pr->box_group[b] : 0];
        for (int c = 0; c < 3; ++c) {
            q[c] = std::min(q[c], (int)pr->box_ijk[3 * b + c]);
            q[3 + c] = std::max(q[3 + c], (int)pr->box_ijk[3 * b + c]);
        }
    }
    double points = 0;
    for (int g = 0; g < G; ++g) {
        if (bb[g][3] < bb[g][0]) continue;      // a scatterer without boxes
        int E[3], L[3];
        for (int c = 0; c < 3; ++c) {
            E[c] = bb[g][3 + c] - bb[g][c] + 1;
            L[c] = E[c] <= 64 ? pad_length(4 * E[c]) : 0;
            if (!L[c]) {
                out.clear();
                return {};
            }
        }
        points += (double)L[0] * L[1] * L[2];
        auto it = std::find_if(out.begin(), out.end(), [&](const ConvClass &c) {
            return c.L[0] == L[0] && c.L[1] == L[1] && c.L[2] == L[2];
        });
        if (it == out.end()) {
            out.emplace_back();
            it = out.end() - 1;
            std::copy(L, L + 3, it->L);
        }
        for (int c = 0; c < 3; ++c) it->E[c] = std::max(it->E[c], E[c]);
        it->group.push_back(g);
        it->lo.push_back({bb[g][0], bb[g][1], bb[g][2]});
    }
    if (points * kPointNs > npairs * kPairNs16 + nblocks * kBlockNs16) mask &= IE_PRECMASK(IE_PREC_FP32);
    if (points * kPointNs > npairs * kPairNs32 + nblocks * kBlockNs32) mask = 0;
    if (!mask) {
        out.clear();
        return {};
    }
    for (auto &c : out) {
        const int64_t ny = 4 * c.E[1], nz = 4 * c.E[2];
        c.a_col = 3 * nz * ny * c.L[0];
        c.b_col = 3 * nz * (int64_t)c.L[1] * c.L[0];
        const int64_t cols = (int64_t)c.group.size() * pr->max_rhs;
        const size_t per = (size_t)(c.a_col + c.b_col) * sizeof(float2);
        c.chunk = (int)std::min<int64_t>(std::min<int64_t>(cols, 16384), std::max<int64_t>(1, kConvWorkspace / per));
    }
    bool even = true;       // with equal boxes every box has enough far sources
    std::vector<int> boxes(G, 0);
    for (int b = 0; b < pr->n_boxes; ++b) ++boxes[pr->box_group ? pr->box_group[b] : 0];
    for (int b = 0; b < pr->n_boxes && even; ++b) {
        const int n = boxes[pr->box_group ? pr->box_group[b] : 0];
        const int near = near_start[b + 1] - near_start[b] + (pr->self_box_mode == 1 ? 1 : 0);
        even = n <= kFarEven * (n - near);
    }
    return {mask, npairs >= kFarPairs && even ? mask : 0u};
}

size_t conv_bytes(const ie_problem *pr, const std::vector<ConvClass> &cl, const ConvUse &use, int64_t nadj,
                  int64_t near_elems) {
    if (cl.empty()) return 0;
    size_t b = 0, a = 0, w = 0, tmp = 0;
    auto add = [&](size_t x) { b += (x + 255) / 256 * 256; };
    for (const auto &c : cl) {
        const size_t K = (size_t)(c.L[0] / 2 + 1) * (c.L[1] / 2 + 1) * (c.L[2] / 2 + 1);
        add(K * 6 * sizeof(float2));
        add(c.group.size() * (size_t)c.E[0] * c.E[1] * c.E[2] * sizeof(int32_t));
        add(c.group.size() * sizeof(int32_t));
        add((size_t)(c.L[0] + c.L[1] + c.L[2]) * sizeof(float2));
        a = std::max(a, (size_t)c.a_col * c.chunk);
        w = std::max(w, (size_t)c.b_col * c.chunk);
        // FP64 octant of one component before and after an axis, freed before the plan returns
        tmp = std::max(tmp, (size_t)(c.L[0] / 2 + 1) * (c.L[1] / 2 + 1) * (c.L[2] / 2 + 1) * 2 * sizeof(double2));
    }
    add(a * sizeof(float2));
    add(w * sizeof(float2));
    b += tmp;
    if (pr->group_nrhs) add((size_t)pr->n_boxes * sizeof(int32_t));
    add(near_elems * sizeof(float2));                                   // short near blocks
    if (!use.far) return b;
    add((size_t)pr->max_rhs * pr->n_boxes * sizeof(double));            // inputs' energies
    add(((size_t)(pr->box_group ? pr->n_groups : 1) + 1) * sizeof(int32_t));
    add(2 * sizeof(int));
    add(2 * (size_t)nadj * sizeof(int32_t));                            // adjacent pairs
    add((size_t)27 * kNU * kNU * sizeof(float2));                       // their masked blocks
    if (pr->prec_mask & (IE_PRECMASK(IE_PREC_BF16X3) | IE_PRECMASK(IE_PREC_FP16X3))) {
        add(2 * (size_t)27 * kTcDispElems * sizeof(uint16_t));
        add(27 * sizeof(int32_t));
    }
    add((size_t)(nadj / 8 + 64) * sizeof(WorkItem) * 4);                // their work lists
    return b;
}

namespace {

ie_status build_khat(ie_plan p, ConvClass &c, cudaStream_t st) {
    const int n[3] = {4 * c.E[0], 4 * c.E[1], 4 * c.E[2]};
    const int64_t K[3] = {c.L[0] / 2 + 1, c.L[1] / 2 + 1, c.L[2] / 2 + 1};
    double2 *t0 = nullptr, *t1 = nullptr;
    double *cs = nullptr;
    // [n_z][n_y][n_x] -> [K_z][n_y][n_x] -> [K_z][K_y][n_x] -> K^
    const size_t s0 = (size_t)std::max<int64_t>((int64_t)n[2] * n[1] * n[0], K[2] * K[1] * n[0]);
    const size_t s1 = (size_t)K[2] * n[1] * n[0];
    const int Lsum = c.L[0] + c.L[1] + c.L[2];
    std::vector<double> h(Lsum);
    std::vector<float2> tw(Lsum);
    for (int ax = 0, o = 0; ax < 3; o += c.L[ax], ++ax)
        for (int j = 0; j < c.L[ax]; ++j) {
            h[o + j] = std::cos(2 * kPi * j / c.L[ax]);
            tw[o + j] = make_float2((float)h[o + j], (float)-std::sin(2 * kPi * j / c.L[ax]));
        }
    IE_CK(cudaMemcpy(c.d_tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice));
    ie_status rc = IE_OK;
    auto body = [&]() -> ie_status {
        IE_TRY(scratch_alloc(&t0, s0, st));
        IE_TRY(scratch_alloc(&t1, s1, st));
        IE_TRY(scratch_alloc(&cs, h.size(), st));
        IE_CK(cudaMemcpyAsync(cs, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice, st));
        const double *ct[3] = {cs, cs + c.L[0], cs + c.L[0] + c.L[1]};
        int comp = 0;
        for (int i = 0; i < 3; ++i)
            for (int j = i; j < 3; ++j, ++comp) {
                const int64_t pts = (int64_t)n[0] * n[1] * n[2];
                conv_green_kernel<<<(unsigned)((pts + 255) / 256), 256, 0, st>>>(p->k, p->eta, p->a / kLattice, n[0], n[1],
                                                                               n[2], i, j, t0);
                IE_CK_LAUNCH();
                // the two sines of an off-diagonal component bring (-j)^2 = -1
                const double scale = (i == j ? 1.0 : -1.0) / ((double)c.L[0] * c.L[1] * c.L[2]);
                auto axis = [&](int ax, const double2 *in, double2 *out, float2 *out32, int64_t inner, int64_t cols) {
                    const dim3 grid((unsigned)((cols + kCt - 1) / kCt), (unsigned)((c.L[ax] / 4 + 1 + kCt - 1) / kCt));
                    conv_axis_kernel<<<grid, kCt * kCt, 0, st>>>(in, out, out32, scale, n[ax], c.L[ax], inner, cols,
                                                                 i != j && (i == ax || j == ax), ct[ax]);
                };
                axis(2, t0, t1, nullptr, (int64_t)n[1] * n[0], (int64_t)n[1] * n[0]);
                IE_CK_LAUNCH();
                axis(1, t1, t0, nullptr, n[0], K[2] * n[0]);
                IE_CK_LAUNCH();
                axis(0, t0, nullptr, reinterpret_cast<float2 *>(c.d_K + (comp / 2) * K[2] * K[1] * K[0]) + comp % 2, 1,
                     K[2] * K[1]);
                IE_CK_LAUNCH();
            }
        return IE_OK;
    };
    rc = body();
    cudaStreamSynchronize(st);      // h is read by the copy
    for (void *q : {(void *)t0, (void *)t1, (void *)cs})
        if (q) cudaFreeAsync(q, st);
    return rc;
}

}  // namespace

ie_status conv_create(ie_plan p, cudaStream_t st) {
    size_t a = 0, w = 0;
    for (auto &c : p->conv) {
        const size_t cells = (size_t)c.E[0] * c.E[1] * c.E[2], ng = c.group.size();
        std::vector<int32_t> slot(cells * ng, -1), cols(ng);
        for (size_t i = 0; i < ng; ++i) {
            const int g = c.group[i];
            cols[i] = p->gnrhs.empty() ? INT_MAX : p->gnrhs[g];
            for (int64_t b = p->gbox[g]; b < p->gbox[g + 1]; ++b) {
                const int32_t *q = &p->ijk[3 * b];
                slot[((i * c.E[2] + (q[2] - c.lo[i][2])) * c.E[1] + (q[1] - c.lo[i][1])) * c.E[0] + (q[0] - c.lo[i][0])] =
                    (int32_t)b;
            }
        }
        IE_TRY(dalloc_t(p, &c.d_slot, slot.size()));
        IE_TRY(dalloc_t(p, &c.d_cols, cols.size()));
        IE_TRY(dalloc_t(p, &c.d_tw, (size_t)c.L[0] + c.L[1] + c.L[2]));
        IE_TRY(dalloc_t(p, &c.d_K, (size_t)(c.L[0] / 2 + 1) * (c.L[1] / 2 + 1) * (c.L[2] / 2 + 1) * 3));
        IE_CK(cudaMemcpy(c.d_slot, slot.data(), slot.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
        IE_CK(cudaMemcpy(c.d_cols, cols.data(), cols.size() * sizeof(int32_t), cudaMemcpyHostToDevice));
        IE_TRY(build_khat(p, c, st));
        a = std::max(a, (size_t)c.a_col * c.chunk);
        w = std::max(w, (size_t)c.b_col * c.chunk);
    }
    if (p->conv.empty()) return IE_OK;
    IE_TRY(dalloc_t(p, &p->d_convA, a));
    IE_TRY(dalloc_t(p, &p->d_convB, w));
    return IE_OK;
}

namespace {

// w[r][b] = sum_u |x_u|^2, a warp per box and column.  The squares are taken at a power of two near
// the box's largest entry, so that neither overflows nor underflows.
__global__ void __launch_bounds__(256) energy_kernel(const float2 *__restrict__ X, int64_t cols, double *__restrict__ w,
                                                     int *__restrict__ form, const int *__restrict__ gate) {
    const bool on = !gate || *gate != 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) form[0] = on, form[1] = 0;
    const int64_t col = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (!on || col >= cols) return;
    const int lane = threadIdx.x & 31;
    float2 x[kNU / 32];
    float m = 0.f;
#pragma unroll
    for (int t = 0; t < kNU / 32; ++t) {
        x[t] = X[col * kNU + lane + 32 * t];
        m = fmaxf(m, fmaxf(fabsf(x[t].x), fabsf(x[t].y)));
    }
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    int e = 0;
    if (m > 0.f && m <= 3.4028235e38f) frexpf(m, &e);   // NaN entries stay in the sum, infinite ones too
    const float down = ldexpf(1.f, -(e / 2)), rest = ldexpf(1.f, e / 2 - e);
    float s = 0.f;
#pragma unroll
    for (int t = 0; t < kNU / 32; ++t) {
        const float a = x[t].x * down * rest, b = x[t].y * down * rest;
        s = fmaf(a, a, fmaf(b, b, s));
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) w[col] = ldexp((double)s, 2 * e);
}

// A CTA takes kFormBoxes boxes of one scatterer and column, a warp four of them, lanes over the
// stored near boxes (27 at most).  Every CTA sums the scatterer's energy itself, in one order.
// Bound by its chain of reads.
constexpr int kFormBoxes = 32;
__global__ void __launch_bounds__(256) choose_form_kernel(const double *__restrict__ w, const int32_t *__restrict__ gbox,
                                                          const int32_t *__restrict__ near_start,
                                                          const int32_t *__restrict__ near_src,
                                                          const int32_t *__restrict__ box_cols, int nbox,
                                                          int *__restrict__ form, const int *__restrict__ gate) {
    if (gate && *gate == 0) return;
    __shared__ double red[8];
    const int b0 = gbox[blockIdx.x], b1 = gbox[blockIdx.x + 1], first = b0 + (int)blockIdx.y * kFormBoxes;
    const int r = blockIdx.z, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (first >= b1 || (box_cols && r >= box_cols[b0])) return;
    const double *wr = w + (int64_t)r * nbox;
    double near[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = min(first + 4 * warp + i, b1 - 1), q = near_start[t] + lane;
        const int src = q < near_start[t + 1] ? near_src[q] : t;
        near[i] = lane == 31 || src != t ? wr[src] : 0.0;       // lane 31 has no entry: the box itself
    }
    double s = 0;
#pragma unroll 8
    for (int b = b0 + threadIdx.x; b < b1; b += 256) s += wr[b];
    for (int o = 16; o; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
#pragma unroll
        for (int i = 0; i < 4; ++i) near[i] += __shfl_xor_sync(0xffffffffu, near[i], o);
    }
    if (lane == 0) red[warp] = s;
    __syncthreads();
    s = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
    bool blocks = !(s == 0 || (s >= kEnergyMin && s <= kEnergyMax));        // NaN too
#pragma unroll
    for (int i = 0; i < 4; ++i) blocks |= !(s <= kFarEven * (s - near[i]));
    if (blocks && lane == 0) form[0] = 0, form[1] = 1;       // one value from every warp
}

}  // namespace

ie_status launch_choose_form(ie_plan p, const float2 *X, int nrhs, cudaStream_t st, const int *gate) {
    const int64_t cols = (int64_t)nrhs * p->nbox;
    energy_kernel<<<(unsigned)((cols + 7) / 8), 256, 0, st>>>(X, cols, p->d_energy, p->d_form, gate);
    IE_CK_LAUNCH();
    int64_t most = 0;
    for (int g = 0; g < p->ngroups; ++g) most = std::max(most, p->gbox[g + 1] - p->gbox[g]);
    const dim3 grid(p->ngroups, (unsigned)((most + kFormBoxes - 1) / kFormBoxes), nrhs);
    choose_form_kernel<<<grid, 256, 0, st>>>(
        p->d_energy, p->d_gbox, p->d_near_start, p->d_near_src, p->d_box_cols, p->nbox, p->d_form, gate);
    IE_CK_LAUNCH();
    return IE_OK;
}

// Bytes the five passes read and write, in L2 or device memory (K^ and the boxes' vectors once each).
int64_t conv_traffic(const ie_plan_s *p, int nrhs) {
    int64_t b = 2 * (int64_t)nrhs * p->nbox * kNU * sizeof(float2);
    for (const auto &c : p->conv) {
        int64_t cols = 0;
        for (int g : c.group) cols += p->gnrhs.empty() ? nrhs : std::min(nrhs, (int)p->gnrhs[g]);
        b += 4 * cols * (c.a_col + c.b_col) * (int64_t)sizeof(float2);
        b += (int64_t)(c.L[0] / 2 + 1) * (c.L[1] / 2 + 1) * (c.L[2] / 2 + 1) * 6 * sizeof(float2);
    }
    return b;
}

// The passes of a small convolution take 3 to 30 us each, and a launch's set-up and ramp about 1.5
// us: they are chained (launch_after).  64 boxes (L = 32) 35 -> 28 us, 16^3 shell (L = 128) 126 ->
// 116, 8 scatterers with four columns 1,099 -> 1,060.  Not from L = 256 on (32^3 shell far 571 ->
// 577 us: the next pass's CTAs hold room beside a long pass) and not under capture (as edges of the
// GMRES cycle's graph: 16^3 shell solve 1,510 -> 1,522 us, 32^3 shell 4,731 -> 4,901).
constexpr int64_t kEarlyPoints = (int64_t)192 * 192 * 192;

ie_status launch_conv(ie_plan p, const float2 *X, float2 *Y, int nrhs, cudaStream_t st, const int *gate) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    IE_CK(cudaStreamIsCapturing(st, &cs));
    const bool capturing = cs != cudaStreamCaptureStatusNone;
    for (const auto &c : p->conv) {
        ConvArgs a;
        a.X = X;
        a.Y = Y;
        a.A = p->d_convA;
        a.B = p->d_convB;
        a.a_col = c.a_col;
        a.b_col = c.b_col;
        a.K = c.d_K;
        a.slot = c.d_slot;
        a.cols = c.d_cols;
        a.twx = c.d_tw;
        a.twy = c.d_tw + c.L[0];
        a.twz = c.d_tw + c.L[0] + c.L[1];
        a.Ex = c.E[0], a.Ey = c.E[1], a.Ez = c.E[2];
        a.Lx = c.L[0], a.Ly = c.L[1], a.Lz = c.L[2];
        a.nbox = p->nbox;
        a.nrhs = nrhs;
        a.gate = gate;
        const bool early = !capturing && (int64_t)a.Lx * a.Ly * a.Lz <= kEarlyPoints;
        const int cols = (int)c.group.size() * nrhs, ny = 4 * a.Ey, nz = 4 * a.Ez;
        for (a.q0 = 0; a.q0 < cols; a.q0 += c.chunk) {
            const unsigned nq = (unsigned)std::min(c.chunk, cols - a.q0);
            auto xgrid = [&](int rows) { return dim3((unsigned)((ny + rows - 1) / rows), (unsigned)nz, nq); };
            const dim3 ygrid(a.Lx / kW, nz, 3 * nq), zgrid(a.Lx / kW, a.Ly, nq);
#define IE_CASE(L, R1, R2) \
    case L: launch_after(early, conv_x_kernel<R1, R2>, xgrid(XTile<R2>::rows), kXThreads, x_smem<R1, R2>(), st, a); break;
            switch (a.Lx) { IE_CONV_SIZES(IE_CASE) }
#undef IE_CASE
            IE_CK_LAUNCH();
#define IE_CASE(L, R1, R2) \
    case L: launch_after(early, conv_y_kernel<R1, R2>, ygrid, kW * R2, y_smem<R1, R2>(), st, a); break;
            switch (a.Ly) { IE_CONV_SIZES(IE_CASE) }
#undef IE_CASE
            IE_CK_LAUNCH();
#define IE_CASE(L, R1, R2, PF, AHEAD, CTAS) \
    case L: launch_after(early, conv_z_kernel<R1, R2, PF, AHEAD, CTAS>, zgrid, kW * R2, z_smem<R1, R2>(), st, a); break;
            switch (a.Lz) { IE_CONV_ZSIZES(IE_CASE) }
#undef IE_CASE
            IE_CK_LAUNCH();
#define IE_CASE(L, R1, R2) \
    case L: launch_after(early, conv_yback_kernel<R1, R2>, ygrid, kW * R2, y_smem<R1, R2>(), st, a); break;
            switch (a.Ly) { IE_CONV_SIZES(IE_CASE) }
#undef IE_CASE
            IE_CK_LAUNCH();
#define IE_CASE(L, R1, R2) \
    case L: launch_after(early, conv_xback_kernel<R1, R2>, xgrid(XTile<R2>::rows), kXThreads, x_smem<R1, R2>(), st, a); break;
            switch (a.Lx) { IE_CONV_SIZES(IE_CASE) }
#undef IE_CASE
            IE_CK_LAUNCH();
        }
    }
    return IE_OK;
}

}  // namespace ie

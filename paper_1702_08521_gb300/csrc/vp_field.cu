// vp_field.cu -- velocity moment, FFT Poisson solver with the 2nd/4th/6th-
// order Green functions (periodic) or doubling-up (isolated), FDA force,
// diagnostics reductions and analytic initial conditions, all on the device.
//
// Precision: f is read as float or double; every sum over velocity space is
// carried in double precision (for float input, short compensated float sums per
// thread -- Knuth's two-sum -- whose values are added in double, then double
// across threads).  Fourier transforms, Green functions
// and forces are double precision throughout.
#include <cmath>
#include <mutex>

#include "vp_internal.cuh"
#include "vp_sum.cuh"

namespace {

constexpr int kBlock = 256;

using vp_sum::PairSum;
using vp_sum::warp_sum;
using vp_sum::widen_any;

// ---- sums over velocity space --------------------------------------------------
//
// Read once, so HBM should set the time; what did was the FP64 pipe (two lanes
// per SM and clock): tree sums of doubles over 256 threads took 20 us for 4096
// points of 1024 cells (67 MB, 10 us of HBM), and the diagnostics' per-cell
// double arithmetic and 64-bit remainders 12.3 ms for 3.1e8 cells (0.18 ms).
// So runs of a few cells are summed as float pairs -- value and error term of
// Knuth's two-sum, products with their exact error from an FMA --, their values
// added in double, and one warp adds the threads' doubles: the density of 3.1e8
// cells 180 us, the diagnostics 0.74 ms (0.93 ms where most cells are subnormal or
// nearly), with the errors of sums in double: 1e-16 of the mass, energy and
// squares.  Whole threads' sums as pairs took 0.80 ms and were off by up to 7e-15.

// ---- density moment ----------------------------------------------------------

// the same sum, for all lanes (or threads) of a point where the value of a pair
// left the float range or a cell is not finite: NaN then, also for an infinite cell
__device__ __noinline__ double part_sum_rare(const float *p, long long n, int t, int nt) {
    double a = 0.0;
    for (long long i = t; i < n; i += nt) {
        const float x = p[i];
        a += (double)x + (double)(x - x);
    }
    return a;
}
__device__ __forceinline__ double part_sum_rare(const double *, long long, int, int) { return 0.0; }

// the lane's (or thread's) part of sum p[0..n): 16-byte loads between the
// unaligned ends, a pair sum whose value goes to a double every 8 cells and whose
// error term is folded then (an error term of n cells rounds by up to n 2^-51)
__device__ __forceinline__ double part_sum(const float *p, long long n, int t, int nt) {
    vp_sum::LongSum a;
    double d = 0.0;
    auto flush = [&]() {
        d += widen_any(a.s);
        a.s = 0.f;
        a.fold();
    };
    auto quad = [&](const float4 &v) {
        a.add(v.x);
        a.add(v.y);
        a.add(v.z);
        a.add(v.w);
    };
    long long head = (long long)((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15) / 4;
    head = head < n ? head : n;
    for (long long i = t; i < head; i += nt) a.add(p[i]);
    const float4 *q = reinterpret_cast<const float4 *>(p + head);
    const long long nq = (n - head) / 4;
    long long i = t;
    for (; i + 3 * nt < nq; i += 4 * nt) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = q[i + k * nt];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            quad(v[k]);
            if (k & 1) flush();
        }
    }
    for (; i < nq; i += nt) {
        quad(q[i]);
        flush();
    }
    for (i = head + 4 * nq + t; i < n; i += nt) a.add(p[i]);
    flush();
    return d + widen_any(a.error());
}

__device__ __forceinline__ double part_sum(const double *p, long long n, int t, int nt) {
    double a = 0.0, b = 0.0;
    long long i = t;
    for (; i + nt < n; i += 2 * nt) {
        a += p[i];
        b += p[i + nt];
    }
    if (i < n) a += p[i];
    return a + b;
}

// WARP: one warp per spatial point (velocity grids of at most kWarpCells
// cells: 4096 points of 1024 cells 20.6 -> 7.1 us), else one block per point
constexpr long long kWarpCells = 2048;

template <typename T, bool WARP>
__global__ void __launch_bounds__(kBlock) k_moment(const T *f, long long NX, long long NV, double dV,
                                                   double *rho) {
    dep_wait();
    dep_launch();
    if (WARP) {
        const long long x = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
        if (x >= NX) return;
        double s = part_sum(f + x * NV, NV, threadIdx.x & 31, 32);
        if (sizeof(T) == 4 && __any_sync(0xffffffffu, !isfinite(s))) s = part_sum_rare(f + x * NV, NV, threadIdx.x & 31, 32);
        s = warp_sum(s);
        if ((threadIdx.x & 31) == 0) rho[x] = s * dV;
    } else {
        // one warp adds the threads' parts: a shuffle tree in every warp would keep
        // the FP64 pipe busy three times as long
        __shared__ double sh[kBlock];
        const T *p = f + (long long)blockIdx.x * NV;
        double s = part_sum(p, NV, threadIdx.x, blockDim.x);
        sh[threadIdx.x] = s;
        if (__syncthreads_or(sizeof(T) == 4 && !isfinite(s))) {
            sh[threadIdx.x] = part_sum_rare(p, NV, threadIdx.x, blockDim.x);
            __syncthreads();
        }
        if (threadIdx.x >= 32) return;
        s = 0.0;
#pragma unroll
        for (int i = 0; i < kBlock / 32; ++i) s += sh[32 * i + threadIdx.x];
        s = warp_sum(s);
        if (threadIdx.x == 0) rho[blockIdx.x] = s * dV;
    }
}

// ---- Fourier transforms of the field solve ---------------------------------------
//
// FP64 is the scarce unit here (two FMA lanes per SM and clock) and a launch
// costs 2.5-4 us, so the solve is few launches that spread the FP64 work:
//   * k_fft_lines transforms B lines of one axis in shared memory (Stockham,
//     radices 4 and 2, odd prime factors as direct sums) with a table of
//     the n roots of unity, read from the context or, for callers without
//     one, computed once per CTA.  The first axis reads rho itself, and the
//     last forward axis multiplies by the Green function and transforms back
//     in the same pass.  Before (radix 2 with a double-precision sincospi per
//     butterfly, direct sums with one per term): 17 us per axis at 64 points
//     and 500 us per axis at 2024 lines of 40 points.
//     The field solve of a 22 x 20 x 23 isolated box: 3.0 -> 0.12 ms; of a
//     64 x 64 periodic box: 84 -> 38 us (serialised launches, cold caches).
//   * k_conv1: in one dimension the solve is a cyclic convolution, n^2 FMAs
//     spread over the chip in one launch.

constexpr int kFftMaxRad = 12;  // factors of an axis length <= 4096

struct FftPlan {
    int n, nr;
    int rad[kFftMaxRad];
    // divisors of the index arithmetic: butterflies per line and distance of a
    // pass, the line length (an integer division is ~150 cycles of latency, and
    // a 64-point line is one warp with nothing to hide it)
    FastDiv fd_m[kFftMaxRad], fd_ns[kFftMaxRad], fd_n;
};

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}

// sum_j x_j exp(sign 2 pi i j k / n) of B lines (line b at x + b n), ping-pong
// between x and y; w[j] = exp(-2 pi i j / n).  Returns the buffer that holds
// the result (natural order); the caller's data must be in place (barrier
// before), and a barrier follows the last pass.
__device__ double2 *fft_lines(double2 *x, double2 *y, const double2 *w, const FftPlan &p, int B, int sign) {
    const int n = p.n;
    const double sg = sign < 0 ? 1.0 : -1.0;  // the table holds the forward roots
    int Ns = 1;
    for (int f = 0; f < p.nr; ++f) {
        const int r = p.rad[f];
        const int m = n / r, ts = m / Ns;  // butterflies per line, table stride of exp(-2 pi i / (Ns r))
        if (r == 4 || r == 2) {
            for (int t = threadIdx.x; t < B * m; t += blockDim.x) {
                const int b = B == 1 ? 0 : (int)fdiv((unsigned)t, p.fd_m[f]), j = t - b * m;
                const int k = (int)fmod_u((unsigned)j, p.fd_ns[f]);
                const double2 *xi = x + b * n + j;
                double2 *yo = y + b * n + (j - k) * r + k;
                auto tw = [&](int q) {
                    const double2 v = w[q * k * ts];
                    return cmul(xi[q * m], make_double2(v.x, sg * v.y));
                };
                if (r == 2) {
                    const double2 a = xi[0], c = tw(1);
                    yo[0] = cadd(a, c);
                    yo[Ns] = csub(a, c);
                } else {
                    const double2 a = xi[0], c = tw(2), d = tw(1), e = tw(3);
                    const double2 s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(d, e), s3 = csub(d, e);
                    const double2 rot = make_double2(sg * s3.y, -sg * s3.x);  // -i (forward) or +i times s3
                    yo[0] = cadd(s0, s2);
                    yo[Ns] = cadd(s1, rot);
                    yo[2 * Ns] = csub(s0, s2);
                    yo[3 * Ns] = csub(s1, rot);
                }
            }
        } else {
            // direct: output o = (block, q, k) sums r inputs with the roots
            // exp(-2 pi i p (k + q Ns) / (Ns r))
            for (int t = threadIdx.x; t < B * n; t += blockDim.x) {
                const int b = B == 1 ? 0 : (int)fdiv((unsigned)t, p.fd_n), o = t - b * n;
                const int blk = o / (Ns * r), kq = o - blk * (Ns * r);
                const double2 *xi = x + b * n + blk * Ns + (int)fmod_u((unsigned)kq, p.fd_ns[f]);
                const int step = kq * ts;  // < n
                double2 a0 = xi[0], a1 = make_double2(0.0, 0.0);
                int idx = 0;
                for (int q = 1; q < r; ++q) {
                    idx += step;
                    idx -= idx >= n ? n : 0;
                    const double2 v = w[idx], u = xi[q * m];
                    const double wy = sg * v.y;
                    a0.x = fma(u.x, v.x, a0.x);
                    a0.y = fma(u.x, wy, a0.y);
                    a1.x = fma(-u.y, wy, a1.x);
                    a1.y = fma(u.y, v.x, a1.y);
                }
                y[t] = cadd(a0, a1);
            }
        }
        __syncthreads();
        double2 *z = x;
        x = y;
        y = z;
        Ns *= r;
    }
    return x;
}

// what a pass of k_fft_lines does with its lines
enum { FFT_FWD = -1, FFT_INV = 1, FFT_CONV = 2 };

struct FftArgs {
    FftPlan p;
    long long lines;      // lines along the axis
    unsigned inner;       // element stride of the axis
    int B;                // lines per CTA (neighbours in the inner index; consecutive lines when inner == 1)
    int mode;
    // first axis (inner == 1): read rho of the box, zero outside it
    const double *rho;
    double bg;
    int nbox[3], m[3], dims;
    // FFT_CONV: real factors, or complex factors times scale
    const double *green;
    const double2 *ghat;
    double scale;
    const double2 *tw;    // n roots of the axis, or NULL: computed in the CTA
};

__global__ void __launch_bounds__(256) k_fft_lines(double2 *a, FftArgs f) {
    extern __shared__ double2 sbuf[];
    const int n = f.p.n, B = f.B;
    double2 *w = sbuf, *x = sbuf + n, *y = x + B * n;
    // first line of the CTA and its element base; lines are base + b (strided
    // axis) or base + b n
    const unsigned tpo = f.inner == 1 ? 1u : (f.inner + B - 1) / B;
    long long base;
    int nb;
    long long l0 = 0;
    if (f.inner == 1) {
        l0 = (long long)blockIdx.x * B;
        nb = (int)(f.lines - l0 < B ? f.lines - l0 : B);
        base = l0 * n;
    } else {
        const unsigned o = blockIdx.x / tpo, c = (blockIdx.x - o * tpo) * B;
        nb = (int)(f.inner - c < (unsigned)B ? f.inner - c : B);
        base = (long long)o * n * f.inner + c;
    }
    if (f.tw) dep_wait();
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        if (f.tw) {
            w[j] = f.tw[j];
        } else {
            double sn, cs;
            sincospi(2.0 * (double)j / (double)n, &sn, &cs);
            w[j] = make_double2(cs, -sn);
        }
    }
    dep_wait();
    dep_launch();
    if (f.rho) {
        // contiguous lines of the padded grid: the line's outer indices, and
        // its row of the box (or a line of zeros)
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) {
            const int b = B == 1 ? 0 : (int)fdiv((unsigned)t, f.p.fd_n), j = t - b * n;
            long long r = l0 + b, row = 0, mul = f.nbox[f.dims - 1];
            bool in = j < f.nbox[f.dims - 1];
            for (int d = f.dims - 2; d >= 0; --d) {
                const int i = (int)((unsigned)r % (unsigned)f.m[d]);
                r = (unsigned)r / (unsigned)f.m[d];
                in = in && i < f.nbox[d];
                row += i * mul;
                mul *= f.nbox[d];
            }
            x[t] = make_double2(in ? f.rho[row + j] - f.bg : 0.0, 0.0);
        }
    } else if (f.inner == 1) {
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) x[t] = a[base + t];
    } else {
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) {
            const int j = nb == 1 ? t : t / nb, b = t - j * nb;
            x[b * n + j] = a[base + (long long)j * f.inner + b];
        }
    }
    __syncthreads();
    double2 *r = fft_lines(x, y, w, f.p, nb, f.mode == FFT_INV ? 1 : -1);
    if (f.mode == FFT_CONV) {
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) {
            int j, b;
            long long g;
            if (f.inner == 1) {
                b = B == 1 ? 0 : (int)fdiv((unsigned)t, f.p.fd_n);
                j = t - b * n;
                g = base + t;
            } else {
                j = nb == 1 ? t : t / nb;
                b = t - j * nb;
                g = base + (long long)j * f.inner + b;
            }
            double2 u = r[b * n + j];
            if (f.green) {
                const double s = f.green[g];
                u = make_double2(u.x * s, u.y * s);
            } else {
                u = cmul(u, f.ghat[g]);
                u = make_double2(u.x * f.scale, u.y * f.scale);
            }
            r[b * n + j] = u;
        }
        __syncthreads();
        r = fft_lines(r, r == x ? y : x, w, f.p, nb, 1);
    }
    if (f.inner == 1) {
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) a[base + t] = r[t];
    } else {
        for (int t = threadIdx.x; t < nb * n; t += blockDim.x) {
            const int j = nb == 1 ? t : t / nb, b = t - j * nb;
            a[base + (long long)j * f.inner + b] = r[b * n + j];
        }
    }
}

// roots of unity w[j] = exp(-2 pi i j / n)
__global__ void k_roots(double2 *__restrict__ w, int n) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double sn, cs;
    sincospi(2.0 * (double)j / (double)n, &sn, &cs);
    w[j] = make_double2(cs, -sn);
}

// One dimension, periodic: phi = g * (rho - bg) and a = k * (rho - bg) are
// cyclic convolutions.  Both kernels sum to zero, so a constant moves nothing, but
// its roundings do (a density 1000 times its variation: phi off by 1.4e-12, by FFT
// 2.7e-14): the middle one of three densities is taken from all in place of the
// background.  The kernels from their spectra (green_k = S / lambda_k
// / n and D_k green_k, D_k the symbol of the FDA): g_j = sum_k green_k cos(2 pi
// j k / n), k_j = sum_k (D green)_k sin(2 pi j k / n).  ker = [g | k].
__global__ void k_conv1_kernels(const double *__restrict__ green, const double *__restrict__ dgreen,
                                const double2 *__restrict__ w, int n, double *__restrict__ ker) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double g = 0.0, k1 = 0.0;
    int idx = 0;
    for (int k = 0; k < n; ++k) {
        const double2 v = w[idx];
        g = fma(green[k], v.x, g);
        k1 = fma(-dgreen[k], v.y, k1);  // the table holds -sin
        idx += j;
        idx -= idx >= n ? n : 0;
    }
    ker[j] = g;
    ker[n + j] = k1;
}

// One warp per output point, lanes over the sum; phi is optional.  n = 64: 1
// launch of ~3 us where load, two transforms, multiply and force took 45 us;
// 4096 points (the largest axis): 2 x 16.8 M FMAs, ~55 us per output array of
// the FP64 pipe, still below the two transforms of one CTA.
constexpr int kConvWarps = 4;
__global__ void __launch_bounds__(32 * kConvWarps) k_conv1(const double *rho, int n, const double *ker, double *phi,
                                                            double *acc) {
    extern __shared__ double srho[];
    dep_wait();
    dep_launch();
    // (the middle one by the numbers' bits on the integer pipe: FP64 comparisons of
    // every thread took 1 us)
    auto key = [](long long b) { return b ^ ((b >> 63) & 0x7fffffffffffffffLL); };  // its own inverse
    const long long *bits = reinterpret_cast<const long long *>(rho);
    const long long k0 = key(bits[0]), k1 = key(bits[n / 3]), k2 = key(bits[2 * (n / 3)]);
    const double mid = __longlong_as_double(key(max(min(k0, k1), min(max(k0, k1), k2))));
    for (int j = threadIdx.x; j < n; j += blockDim.x) srho[j] = rho[j] - mid;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kConvWarps + (threadIdx.x >> 5);
    if (i >= n) return;
    double s0 = 0.0, s1 = 0.0, p0 = 0.0;
    const double *g = ker, *k = ker + n;
    int j = lane;
#pragma unroll 4
    for (; j + 32 < n; j += 64) {
        int d0 = i - j, d1 = d0 - 32;
        d0 += d0 < 0 ? n : 0;
        d1 += d1 < 0 ? n : 0;
        s0 = fma(k[d0], srho[j], s0);
        s1 = fma(k[d1], srho[j + 32], s1);
        if (phi) p0 = fma(g[d1], srho[j + 32], fma(g[d0], srho[j], p0));
    }
    if (j < n) {
        int d0 = i - j;
        d0 += d0 < 0 ? n : 0;
        s0 = fma(k[d0], srho[j], s0);
        if (phi) p0 = fma(g[d0], srho[j], p0);
    }
    s0 = warp_sum(s0 + s1);
    if (phi) p0 = warp_sum(p0);
    if (lane == 0) {
        acc[i] = s0;
        if (phi) phi[i] = p0;
    }
}

// phi (box) and accel = -grad phi by the 2/4/6-point FDA (Eqs. C9-C11),
// reading the potential of the m-periodic grid (m = box for periodic,
// m = 2 box for doubling-up) with cyclic indices.  32-bit index arithmetic
// (the grid is below 2^31 points) and the factor 1 / (den h) from the host:
// 15 -> 4 us at 16^3 points, where 64-bit remainders and FP64 divisions set
// the time.
struct Fda {
    double c[4];  // c[k] multiplies (phi_{i+k} - phi_{i-k}), k = 1..3
    double den;
};

struct ForceArgs {
    unsigned NX;
    FastDiv nb1, nb2;      // box sizes of the second and third axis
    int m[3];              // transformed grid
    int dims, npts;
    double c[4];
    double inv[3];         // -1 / (den h) per axis
};

__global__ void __launch_bounds__(kBlock) k_force(const double2 *a, double *phi,
                                                  double *acc, ForceArgs f) {
    dep_wait();
    dep_launch();
    const unsigned x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= f.NX) return;
    int i[3];
    unsigned q = fdiv(x, f.nb2);
    i[2] = (int)(x - q * f.nb2.d);
    i[0] = (int)fdiv(q, f.nb1);
    i[1] = (int)(q - (unsigned)i[0] * f.nb1.d);
    // axes beyond dims have one cell: strides of the transformed grid
    const int st[3] = {f.m[1] * f.m[2], f.m[2], 1};
    const double2 *p = a + ((long long)i[0] * st[0] + (long long)i[1] * st[1] + i[2]);
    if (phi) phi[x] = p->x;
    for (int d = 0; d < f.dims; ++d) {
        double g = 0.0;
        for (int k = 1; k <= f.npts; ++k) {
            int up = i[d] + k, dn = i[d] - k;
            while (up >= f.m[d]) up -= f.m[d];
            while (dn < 0) dn += f.m[d];
            g = fma(f.c[k], p[(long long)(up - i[d]) * st[d]].x - p[(long long)(dn - i[d]) * st[d]].x, g);
        }
        acc[(long long)d * f.NX + x] = g * f.inv[d];
    }
}

// ---- diagnostics -----------------------------------------------------------

// Weights of the kinetic energy: |v|^2 over the axes before the last (one entry
// per velocity row) and over the last axis, divided by a power of two near the
// largest so that the float pairs neither overflow nor lose their low part.
struct WPair {
    float hi, lo;
};

struct VWeights {
    double lo[3], h[3];
    int n[3];
    int dv;
    double unit;  // the power of two
};

__device__ __forceinline__ void put_weight(WPair *w, double v) {
    w->hi = (float)v;
    w->lo = (float)(v - (double)w->hi);
}
__device__ __forceinline__ void put_weight(double *w, double v) { *w = v; }

template <typename W>
__global__ void k_vweights(VWeights g, long long rows, W *__restrict__ wrow, W *__restrict__ wlast) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int last = g.dv - 1;
    if (t < rows) {
        long long r = t;
        double v2 = 0.0;
        for (int d = last - 1; d >= 0; --d) {
            const double vc = g.lo[d] + ((double)(r % g.n[d]) + 0.5) * g.h[d];
            r /= g.n[d];
            v2 += vc * vc;
        }
        put_weight(wrow + t, v2 / g.unit);
    }
    if (t < g.n[last]) {
        const double vc = g.lo[last] + ((double)t + 0.5) * g.h[last];
        put_weight(wlast + t, vc * vc / g.unit);
    }
}

// the per-cell sums of one thread
template <typename T>
struct DiagSum;

template <>
struct DiagSum<float> {
    using W = WPair;
    // A thread's sums of its cells times `scale`, 2^100 until it meets one of 2^-40,
    // then 1 (with the sums so far): no product of scaled cells, nor its error term,
    // leaves the float range, and what underflows in those of small cells beside a
    // larger one is below 2^-69 of the sums.  Fallen tails of a distribution are full
    // of such cells; sending them through FP64 took 5.9 ms for 3.1e8 cells.
    vp_sum::LongSum m0;
    vp_sum::ProductSum m2;
    vp_sum::SquareSum l2;
    PairSum neg;
    // the values of the pairs so far: cells, weighted cells, negative cells, squares
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    float mn = INFINITY, mx = -INFINITY, scale = kUp;
    bool huge = false, bad = false;  // a cell above 2^60: the point is summed again in double
    bool held = false;               // the doubles hold sums
    static constexpr float kUp = 0x1p100f, kPlain = 0x1p-40f, kHuge = 0x1p60f;
    static constexpr double kDown = 0x1p-100;
    __device__ __forceinline__ void any(float x, const W &w) {
        m2.add_product(x, w.hi);
        m2.q = fmaf(x, w.lo, m2.q);
    }
    // to the scale 1 (mostly before any cell that is not empty)
    __device__ __forceinline__ void unscale() {
        scale = 1.f;
        if (l2.s == 0.f && !held) return;
        flush();
        flush_errors();
        v[0] *= kDown;
        v[1] *= kDown;
        v[2] *= kDown;
        v[3] *= kDown * kDown;
        m0 = vp_sum::LongSum();
        m2 = vp_sum::ProductSum();
        l2 = vp_sum::SquareSum();
        neg = PairSum();
    }
    __device__ __forceinline__ void cell(float x, const W &w, const W *w2) {
        mn = fminf(mn, x);
        mx = fmaxf(mx, x);
        if (!(fabsf(x) <= kHuge)) huge = true;
        if (fabsf(x) >= kPlain && scale != 1.f) unscale();
        const float y = x * scale;
        m0.add(y);
        any(y, w);
        if (w2) any(y, *w2);
        l2.add_square(y);
        if (x < 0.f) neg.add(y);
    }
    // four cells of one index of the last axis
    __device__ __forceinline__ void cells(const float (&x)[4], const W (&w)[4]) {
        const float lo = fminf(fminf(x[0], x[1]), fminf(x[2], x[3])), hi = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
        mn = fminf(mn, lo);
        mx = fmaxf(mx, hi);
        const float size = fmaxf(hi, -lo);
        // (x - x: not a number for cells that are not finite, which the extrema skip)
        const float z = ((x[0] - x[0]) + (x[1] - x[1])) + ((x[2] - x[2]) + (x[3] - x[3]));
        if (!(size + z <= kHuge)) huge = true;
        if (size == 0.f) return;
        if (size >= kPlain && scale != 1.f) unscale();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float y = x[k] * scale;
            m0.add(y);
            any(y, w[k]);
            l2.add_square(y);
            if (k == 1) l2.fold();
        }
        if (lo < 0.f)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (x[k] < 0.f) neg.add(x[k] * scale);
        fold();
    }
    // every four cells: the error terms
    __device__ __forceinline__ void fold() {
        m0.fold();
        m2.fold();
        l2.fold();
    }
    // the pairs' values to the doubles, every 16 cells (the errors of a pair sum
    // grow with its value)
    __device__ __forceinline__ void flush() {
        held = true;
        v[0] += widen_any(m0.s);
        v[1] += widen_any(m2.s);
        v[3] += widen_any(l2.s);
        m0.s = m2.s = l2.s = 0.f;
        if (neg.s != 0.f) {
            v[2] += widen_any(neg.s);
            neg.s = 0.f;
        }
    }
    __device__ __forceinline__ void flush_errors() {
        v[0] += widen_any(m0.error());
        v[1] += widen_any(m2.error());
        v[3] += widen_any(l2.error()) + widen_any(l2.product_error());
        if (neg.e != 0.f) v[2] += widen_any(neg.e);
    }
    // the end of a thread's sums, its cells of one index of the last axis with its
    // weight (NULL: weighed already)
    __device__ __forceinline__ void finish(const W *w) {
        if (scale != 1.f) unscale();
        if (held) {
            flush();
            flush_errors();
        } else {
            v[0] = widen_any(m0.s) + widen_any(m0.error());
            v[1] = widen_any(m2.s) + widen_any(m2.error());
            v[3] = widen_any(l2.s) + (widen_any(l2.error()) + widen_any(l2.product_error()));
            if (neg.s != 0.f) v[2] = widen_any(neg.s) + widen_any(neg.e);
        }
        if (w) v[1] = fma(widen_any(w->hi) + widen_any(w->lo), v[0], v[1]);
    }
};

// the sums of a point with cells that the float pairs cannot hold, in double
// (out of line: its arithmetic would otherwise be predicated into every cell)
__device__ __noinline__ void diag_in_double(const float *p, long long NV, int nlast, const WPair *wrow,
                                            const WPair *wlast, double (&v)[4], bool &bad) {
    for (int k = 0; k < 4; ++k) v[k] = 0.0;
    for (long long i = threadIdx.x; i < NV; i += blockDim.x) {
        const double x = (double)p[i];
        const long long r = i / nlast;
        const WPair a = wrow[r], b = wlast[i - r * nlast];
        if (!isfinite(x)) bad = true;
        v[0] += x;
        v[1] = fma(x, ((double)a.hi + (double)a.lo) + ((double)b.hi + (double)b.lo), v[1]);
        if (x < 0.0) v[2] += x;
        v[3] = fma(x, x, v[3]);
    }
}
__device__ __forceinline__ void diag_in_double(const double *, long long, int, const double *, const double *,
                                               double (&)[4], bool &) {}

template <>
struct DiagSum<double> {
    using W = double;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    double mn = INFINITY, mx = -INFINITY;
    bool bad = false;
    static constexpr bool huge = false;
    __device__ __forceinline__ void cell(double x, const W &w, const W *w2) {
        mn = fmin(mn, x);
        mx = fmax(mx, x);
        if (!isfinite(x)) bad = true;
        v[0] += x;
        v[1] = fma(x, w2 ? w + *w2 : w, v[1]);
        v[3] = fma(x, x, v[3]);
        if (x < 0.0) v[2] += x;
    }
    __device__ __forceinline__ void cells(const double (&x)[4], const W (&w)[4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) cell(x[k], w[k], nullptr);
    }
    __device__ __forceinline__ void fold() {}
    __device__ __forceinline__ void flush() {}
    __device__ __forceinline__ void finish(const W *w) {
        if (w) v[1] = fma(v[0], *w, v[1]);
    }
};

__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double vmin(double a, double b) { return fmin(a, b); }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }

// Sums of one spatial point's cells and its density.  A thread keeps one index
// of the last axis where that axis fits the block (its weight is then applied
// once, to the thread's sum) and walks the rows; longer last axes are walked
// cell by cell with both weights.
template <typename T>
__global__ void __launch_bounds__(kBlock, 4) k_diag_part(const T *f, long long NV, int nlast, FastDiv fd_last,
                                                      const typename DiagSum<T>::W *wrow,
                                                      const typename DiagSum<T>::W *wlast, double unit,
                                                      double dV, double *part,
                                                      double *rho, int *bad) {
    __shared__ double sh[4][kBlock];
    __shared__ T smin[32], smax[32];
    dep_wait();
    dep_launch();
    const T *p = f + (long long)blockIdx.x * NV;
    DiagSum<T> q;
    if (nlast <= (int)blockDim.x) {
        const int nr = (int)fdiv(blockDim.x, fd_last);  // rows at a time
        const int r0 = (int)fdiv(threadIdx.x, fd_last), j = threadIdx.x - r0 * nlast;
        if (r0 < nr) {
            const long long rows = NV / nlast;
            const T *c = p + threadIdx.x;
            const int step = nr * nlast;
            // four cells and weights in flight
            long long r = r0;
            for (int it = 1; r + 3 * nr < rows; r += 4 * nr, ++it) {
                T x[4];
                typename DiagSum<T>::W w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[k] = *c;
                    w[k] = wrow[r + k * nr];
                    c += step;
                }
                q.cells(x, w);
                if ((it & 3) == 0) q.flush();
            }
            for (; r < rows; r += nr) {
                q.cell(*c, wrow[r], nullptr);
                c += step;
            }
            q.finish(wlast + j);
        }
    } else {
        for (long long v = threadIdx.x, it = 1; v < NV; v += 4 * (int)blockDim.x, ++it) {
            T x[4];
            typename DiagSum<T>::W w[4], w2[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const long long i = v + k * (int)blockDim.x;
                if (i < NV) {
                    const long long r = NV < (1LL << 32) ? (long long)fdiv((unsigned)i, fd_last) : i / nlast;
                    x[k] = p[i];
                    w[k] = wrow[r];
                    w2[k] = wlast[i - r * nlast];
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (v + k * (int)blockDim.x < NV) q.cell(x[k], w[k], &w2[k]);
            q.fold();
            if ((it & 3) == 0) q.flush();
        }
        q.finish(nullptr);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (sizeof(T) == 4 && __syncthreads_or(q.huge)) diag_in_double(p, NV, nlast, wrow, wlast, q.v, q.bad);
    if (q.bad) atomicExch(bad, 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) sh[k][threadIdx.x] = q.v[k];
    T mn = q.mn, mx = q.mx;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = vmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = vmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        smin[threadIdx.x >> 5] = mn;
        smax[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    // one warp per sum (a shuffle tree per sum in every warp keeps the FP64 pipe
    // busy three times as long)
    if (warp >= 4) return;
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += sh[warp][32 * i + lane];
    t = warp_sum(t);
    if (lane) return;
    double *o = part + (long long)blockIdx.x * 6;
    if (warp == 0) {
        o[0] = t;
        rho[blockIdx.x] = t * dV;
        for (int k = 1; k < nw; ++k) {
            mn = vmin(mn, smin[k]);
            mx = vmax(mx, smax[k]);
        }
        o[4] = (double)mn;
        o[5] = (double)mx;
    } else {
        o[warp] = warp == 1 ? 0.5 * unit * t : t;
    }
}

// Field terms and the sums over space: every block reduces 256 points, the
// last one to finish the blocks' results (in their order).  One block for all
// points took 189 us at 10120 points, with a double-precision sincospi each.
constexpr int kDiagSums = 8;

__global__ void __launch_bounds__(kBlock) k_diag_final(const double *part,
                                                       const double *rho,
                                                       const double *phi,
                                                       const double *acc, long long NX, int dims, int n1,
                                                       long long rest, int mode, const double2 *roots,
                                                       int root_step, double bg, double dX, double dV,
                                                       double *blk, unsigned *counter,
                                                       double *out) {
    // eight sums and the extrema over the block's 256 points: one warp per sum
    // reads its column of the shared copy (a shuffle tree per sum and warp
    // keeps the FP64 pipe busy 3x longer: 10.3 us for 256 points)
    __shared__ double sv[kDiagSums][kBlock], mm[2][kBlock], res[kDiagSums + 2];
    __shared__ bool last;
    double v[kDiagSums] = {0, 0, 0, 0, 0, 0, 0, 0};
    double mn = INFINITY, mx = -INFINITY;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto reduce = [&]() {
#pragma unroll
        for (int k = 0; k < kDiagSums; ++k) sv[k][threadIdx.x] = v[k];
        mm[0][threadIdx.x] = mn;
        mm[1][threadIdx.x] = mx;
        __syncthreads();
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < kBlock / 32; ++i) t += sv[warp][32 * i + lane];
        t = warp_sum(t);
        if (lane == 0) res[warp] = t;
        if (warp < 2) {
            double e = mm[warp][lane];
#pragma unroll
            for (int i = 1; i < kBlock / 32; ++i) {
                const double o = mm[warp][32 * i + lane];
                e = warp ? fmax(e, o) : fmin(e, o);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double u = __shfl_xor_sync(0xffffffffu, e, o);
                e = warp ? fmax(e, u) : fmin(e, u);
            }
            if (lane == 0) res[kDiagSums + warp] = e;
        }
        __syncthreads();
    };
    static_assert(kDiagSums == kBlock / 32, "one warp per sum");
    dep_wait();
    dep_launch();
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (x < NX) {
        const double *q = part + x * 6;
        v[0] = q[0];
        v[1] = q[1];
        v[2] = q[2];
        v[3] = q[3];
        mn = q[4];
        mx = q[5];
        double fe = 0.0;
        for (int d = 0; d < dims; ++d) fe = fma(acc[d * NX + x], acc[d * NX + x], fe);
        v[4] = 0.5 * fe;
        v[5] = 0.5 * (rho[x] - bg) * phi[x];
        // exp(-2 pi i mode j_1 / n_1), mode in [0, n_1)
        const unsigned k = (unsigned)(((unsigned long long)mode * ((unsigned)x / (unsigned)rest)) % (unsigned)n1);
        const double2 w = roots[k * root_step];
        v[6] = acc[x] * w.x;
        v[7] = acc[x] * w.y;
    }
    reduce();
    if (gridDim.x > 1) {
        double *b = blk + (long long)blockIdx.x * (kDiagSums + 2);
        if (threadIdx.x < kDiagSums + 2) b[threadIdx.x] = res[threadIdx.x];
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            last = atomicAdd(counter, 1u) == gridDim.x - 1;
            if (last) *counter = 0;  // ready for the next launch of the stream
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
#pragma unroll
        for (int k = 0; k < kDiagSums; ++k) v[k] = 0.0;
        mn = INFINITY;
        mx = -INFINITY;
        for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) {
            const double *q = blk + (long long)i * (kDiagSums + 2);
            for (int k = 0; k < kDiagSums; ++k) v[k] += __ldcg(q + k);
            mn = fmin(mn, __ldcg(q + kDiagSums));
            mx = fmax(mx, __ldcg(q + kDiagSums + 1));
        }
        reduce();
    }
    if (threadIdx.x == 0) {
        out[0] = res[0] * dX * dV;
        out[1] = res[1] * dX * dV;
        out[2] = res[4] * dX;
        out[3] = res[5] * dX;
        out[4] = res[kDiagSums];
        out[5] = res[kDiagSums + 1];
        out[6] = 2.0 / (double)NX * sqrt(res[6] * res[6] + res[7] * res[7]);
        out[7] = (res[0] - 2.0 * res[2]) * dX * dV;  // sum |f|
        out[8] = res[3] * dX * dV;
    }
}

// ---- initial conditions ------------------------------------------------------

struct IcArgs {
    int kind, dims;
    int nx[3], nv[3];
    double xlo[3], hx[3], vlo[3], hv[3], xc[3];
    double p[8];
    long long NV;
};

template <typename T>
__global__ void k_init(T *__restrict__ f, long long ncell, IcArgs a) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ncell) return;
    long long xi = t / a.NV, vi = t % a.NV;
    double xs[3] = {0, 0, 0}, vs[3] = {0, 0, 0};
    for (int d = a.dims - 1; d >= 0; --d) {
        xs[d] = a.xlo[d] + ((double)(xi % a.nx[d]) + 0.5) * a.hx[d];
        xi /= a.nx[d];
        vs[d] = a.vlo[d] + ((double)(vi % a.nv[d]) + 0.5) * a.hv[d];
        vi /= a.nv[d];
    }
    const double kPi = 3.141592653589793238462643383279502884;
    double val = 0.0;
    if (a.kind == VP_IC_LANDAU) {
        const double alpha = a.p[0], sig = a.p[4], amp = a.p[5];
        double sp = 1.0, g = 1.0;
        for (int d = 0; d < a.dims; ++d) {
            sp += alpha * cos(a.p[1 + d] * xs[d]);
            g *= exp(-vs[d] * vs[d] / (2.0 * sig * sig)) / sqrt(2.0 * kPi * sig * sig);
        }
        val = amp * sp * g;
    } else if (a.kind == VP_IC_TWOSTREAM) {
        double v2 = 0.0;
        for (int d = 0; d < a.dims; ++d) v2 += vs[d] * vs[d];
        val = vs[0] * vs[0] * exp(-0.5 * v2) / pow(2.0 * kPi, 0.5 * a.dims) *
              (1.0 + a.p[0] * cos(a.p[1] * xs[0]));
    } else if (a.kind == VP_IC_PLUMMER) {
        const double G = a.p[0], M = a.p[1], b = a.p[2];
        double r2 = 0.0, v2 = 0.0;
        for (int d = 0; d < 3; ++d) {
            r2 += (xs[d] - a.xc[d]) * (xs[d] - a.xc[d]);
            v2 += vs[d] * vs[d];
        }
        const double E = 0.5 * v2 - G * M / sqrt(r2 + b * b);
        // isotropic Plummer model: F(E) = 24 sqrt(2) a^2 / (7 pi^3 G^5 M^4) (-E)^(7/2)
        val = E < 0.0 ? 24.0 * sqrt(2.0) * b * b / (7.0 * kPi * kPi * kPi * pow(G, 5.0) * pow(M, 4.0)) *
                            pow(-E, 3.5)
                      : 0.0;
    } else if (a.kind == VP_IC_SPHERE) {
        // uniform sphere of mass M and radius 2R about the box centre with a
        // Maxwellian of sigma^2 = G M / (20 R) (Eq. 77, Sec. 3.4)
        const double G = a.p[0], M = a.p[1], R = a.p[2];
        const double rho0 = M / (4.0 * kPi * (8.0 * R * R * R) / 3.0);
        const double s2 = G * M / (20.0 * R);
        double r2 = 0.0, v2 = 0.0;
        for (int d = 0; d < 3; ++d) {
            r2 += (xs[d] - a.xc[d]) * (xs[d] - a.xc[d]);
            v2 += vs[d] * vs[d];
        }
        val = r2 < 4.0 * R * R ? rho0 * exp(-v2 / (2.0 * s2)) / pow(2.0 * kPi * s2, 1.5) : 0.0;
    } else {
        const int shape = (int)a.p[0];
        if (shape == 0) {
            val = 1.0;
            for (int d = 0; d < a.dims; ++d)
                if (!(xs[d] >= 0.25 && xs[d] <= 0.75)) val = 0.0;
        } else if (shape == 1) {
            val = 1.0;
            for (int d = 0; d < a.dims; ++d) val += sin(2.0 * kPi * xs[d]) / a.dims;
        } else {
            for (int d = 0; d < a.dims; ++d) {
                const double s = sin(4.0 * kPi * xs[d]);
                val += s * s * s * s;
            }
        }
    }
    f[t] = (T)val;
}

inline unsigned nblk(long long n, int b) { return (unsigned)((n + b - 1) / b); }

// radices of an axis of n points: 4s first (fewest FP64 operations), then 2,
// then the odd primes
FftPlan fft_plan(int n) {
    FftPlan p{};
    p.n = n;
    int r = n;
    while (r % 4 == 0) {
        p.rad[p.nr++] = 4;
        r /= 4;
    }
    for (int q = 2; r > 1; q += q == 2 ? 1 : 2) {
        if ((long long)q * q > r) q = r;
        while (r % q == 0) {
            p.rad[p.nr++] = q;
            r /= q;
        }
    }
    int Ns = 1;
    for (int f = 0; f < p.nr; ++f) {
        p.fd_m[f] = make_fastdiv((unsigned)(n / p.rad[f]));
        p.fd_ns[f] = make_fastdiv((unsigned)Ns);
        Ns *= p.rad[f];
    }
    p.fd_n = make_fastdiv((unsigned)n);
    return p;
}

// launch the transform of one axis of the row-major grid m[0..dims)
struct FftLaunch {
    FftArgs f;
    unsigned blocks;
    int threads;
    size_t smem;
};

FftLaunch fft_axis(const int *m, int dims, int axis, int mode, const double2 *tw, int sms) {
    FftLaunch l{};
    FftArgs &f = l.f;
    f.p = fft_plan(m[axis]);
    f.mode = mode;
    f.tw = tw;
    f.dims = dims;
    long long total = 1, inner = 1;
    for (int d = 0; d < dims; ++d) total *= m[d];
    for (int d = axis + 1; d < dims; ++d) inner *= m[d];
    const int n = m[axis];
    f.lines = total / n;
    f.inner = (unsigned)inner;
    // up to four neighbouring lines per CTA (64-byte rows on a strided axis), as many
    // as leave two CTAs per SM
    int B = f.lines >= 8LL * sms ? 4 : (f.lines >= 4LL * sms ? 2 : 1);
    while (B > 1 && (size_t)(1 + 2 * B) * n * sizeof(double2) > 96 * 1024) B /= 2;
    f.B = B;
    l.blocks = inner == 1 ? (unsigned)((f.lines + B - 1) / B)
                          : (unsigned)(f.lines / inner * ((inner + B - 1) / B));
    const int work = B * (f.p.nr && f.p.rad[0] == 4 ? n / 4 : n / 2);
    l.threads = work < 32 ? 32 : (work > 256 ? 256 : (work + 31) / 32 * 32);
    l.smem = (size_t)(1 + 2 * B) * n * sizeof(double2);
    return l;
}

int fft_launch(cudaStream_t st, double2 *buf, const FftLaunch &l) {
    vp_launch_dep(k_fft_lines, l.blocks, l.threads, l.smem, st, buf, l.f);
    return 1;
}

constexpr int kFftSmem = 3 * 4096 * (int)sizeof(double2);  // table and two buffers of the longest axis

Fda fda_coeffs(int order) {
    // central differences of Eqs. (C9)-(C11): sum_k c_k (phi_{i+k} - phi_{i-k}) / (den h)
    Fda f{};
    if (order == 2) {
        f.c[1] = 1.0;
        f.den = 2.0;
    } else if (order == 4) {
        f.c[1] = 8.0;
        f.c[2] = -1.0;
        f.den = 12.0;
    } else {
        f.c[1] = 45.0;
        f.c[2] = -9.0;
        f.c[3] = 1.0;
        f.den = 60.0;
    }
    return f;
}

ForceArgs force_args(const vp_grid &g, const int *m, long long NX) {
    const Fda fd = fda_coeffs(g.pois_order);
    ForceArgs f{};
    f.NX = (unsigned)NX;
    f.dims = g.dx;
    f.npts = g.pois_order / 2;
    f.nb1 = make_fastdiv(g.dx > 1 ? (unsigned)g.nx[1] : 1u);
    f.nb2 = make_fastdiv(g.dx > 2 ? (unsigned)g.nx[2] : 1u);
    for (int k = 0; k < 4; ++k) f.c[k] = fd.c[k];
    for (int d = 0; d < 3; ++d) {
        f.m[d] = d < g.dx ? m[d] : 1;
        f.inv[d] = d < g.dx ? -1.0 / (fd.den * ((g.xhi[d] - g.xlo[d]) / g.nx[d])) : 0.0;
    }
    return f;
}

}  // namespace

// ---- setup: Green functions -----------------------------------------------------

// Eigenvalue of the periodic discrete Laplacian stencil (Eqs. C1, C5, C6)
// for theta = k h, written from its coefficients: with the symmetric stencil
// (b_0, b_1, b_2, b_3) / den the eigenvalue is -(4/den) sum_m b_m sin^2(m theta / 2).
static double stencil_eig(int order, double theta) {
    double b[4] = {0, 0, 0, 0}, den = 1.0;
    if (order == 2) {
        b[1] = 1.0;
    } else if (order == 4) {
        b[1] = 16.0;
        b[2] = -1.0;
        den = 12.0;
    } else {
        b[1] = 270.0;
        b[2] = -27.0;
        b[3] = 2.0;
        den = 180.0;
    }
    double s = 0.0;
    for (int mm = 1; mm <= 3; ++mm) {
        const double q = sin(0.5 * mm * theta);
        s += b[mm] * q * q;
    }
    return -4.0 * s / den;
}

// mean of 1/r over a cube of side 1 about its centre: 24 pyramids with apex
// at the centre give 3 * int_0^1 int_0^1 (1 + u^2 + v^2)^(-1/2) du dv, here by
// composite Gauss-Legendre quadrature (the integrand is smooth).
static double cube_inv_r_mean() {
    const double xg[5] = {-0.9061798459386640, -0.5384693101056831, 0.0, 0.5384693101056831,
                          0.9061798459386640};
    const double wg[5] = {0.2369268850561891, 0.4786286704993665, 0.5688888888888889,
                          0.4786286704993665, 0.2369268850561891};
    const int nsub = 40;
    double s = 0.0;
    for (int a = 0; a < nsub; ++a)
        for (int i = 0; i < 5; ++i) {
            const double u = (a + 0.5 * (xg[i] + 1.0)) / nsub;
            for (int b2 = 0; b2 < nsub; ++b2)
                for (int j = 0; j < 5; ++j) {
                    const double v = (b2 + 0.5 * (xg[j] + 1.0)) / nsub;
                    s += wg[i] * wg[j] / sqrt(1.0 + u * u + v * v);
                }
        }
    return 3.0 * s / (4.0 * nsub * nsub);
}

static int diag_weights(vp_ctx *c);

FieldSizes vp_field_sizes(const vp_ctx *c) {
    const vp_grid &g = c->g;
    const bool iso = g.poisson == VP_POIS_ISOLATED, conv = !iso && g.dx == 1;
    FieldSizes s{};
    for (int d = 0; d < g.dx; ++d) s.roots += sizeof(double2) * (iso ? 2 : 1) * g.nx[d];
    s.green = iso ? 0 : sizeof(double) * (conv ? 2 : 1) * c->NX;
    s.conv = conv ? sizeof(double) * 2 * c->NX : 0;
    const int nlast = g.nv[g.dv - 1];
    s.weights = sizeof(double) * (c->NV / nlast + nlast);
    s.diagblk = sizeof(double) * (kDiagSums + 2) * nblk(c->NX, kBlock);
    return s;
}

int vp_field_setup(vp_ctx *c) {
    const vp_grid &g = c->g;
    const int rcw = diag_weights(c);
    if (rcw) return rcw;
    VP_CUDA_TRY(c, cudaFuncSetAttribute(k_fft_lines, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmem));
    const int D = g.dx;
    const bool iso = g.poisson == VP_POIS_ISOLATED;
    long long nroot = 0;
    for (int d = 0; d < D; ++d) {
        const int m = iso ? 2 * g.nx[d] : g.nx[d];
        c->roots[d] = c->d_roots + nroot;
        k_roots<<<nblk(m, kBlock), kBlock>>>(c->d_roots + nroot, m);
        nroot += m;
    }
    VP_CUDA_TRY(c, cudaGetLastError());
    if (g.poisson == VP_POIS_PERIODIC) {
        c->MT = c->NX;
        for (int d = 0; d < 3; ++d) c->m[d] = d < D ? g.nx[d] : 1;
        // one dimension: the spectrum of the convolution kernels, [green | D green]
        const long long ng = D == 1 ? 2 * c->NX : c->NX;
        double *h_g = (double *)malloc(sizeof(double) * ng);
        if (!h_g) return vp_fail(c, VP_ENOMEM, "host allocation failed");
        const Fda fd = fda_coeffs(g.pois_order);
        for (long long x = 0; x < c->NX; ++x) {
            long long r = x;
            int allzero = 1;
            double lam = 0.0;
            for (int d = D - 1; d >= 0; --d) {
                const long long nk = r % g.nx[d];
                r /= g.nx[d];
                if (nk) allzero = 0;
                const double h = (g.xhi[d] - g.xlo[d]) / g.nx[d];
                lam += stencil_eig(g.pois_order, 2.0 * M_PI * (double)nk / (double)g.nx[d]) / (h * h);
            }
            // phi_hat = S rho_hat / lambda; the inverse transform's 1/NX is folded in
            h_g[x] = allzero ? 0.0 : g.coupling / lam / (double)c->NX;
            if (D == 1) {
                // a = -grad phi: the FDA's symbol is i D, D = sum 2 c_m sin(m theta) / (den h)
                double sym = 0.0;
                for (int mm = 1; mm <= g.pois_order / 2; ++mm)
                    sym += 2.0 * fd.c[mm] * sin(2.0 * M_PI * (double)((mm * x) % g.nx[0]) / (double)g.nx[0]);
                h_g[c->NX + x] = h_g[x] * (sym / (fd.den * ((g.xhi[0] - g.xlo[0]) / g.nx[0])));
            }
        }
        const cudaError_t e = cudaMemcpy(c->d_green, h_g, sizeof(double) * ng, cudaMemcpyHostToDevice);
        free(h_g);
        VP_CUDA_TRY(c, e);
        if (D == 1) {
            const int n = g.nx[0];
            k_conv1_kernels<<<nblk(n, 64), 64>>>(c->d_green, c->d_green + n, c->d_roots, n, c->d_conv);
            VP_CUDA_TRY(c, cudaGetLastError());
        } else {
            VP_CUDA_TRY(c, cudaMalloc(&c->d_fft, sizeof(double2) * c->MT));
        }
        // the tables were made on the legacy stream, which the context's need not wait for
        VP_CUDA_TRY(c, cudaStreamSynchronize(cudaStreamLegacy));
        return VP_OK;
    }
    // isolated: doubling-up with the real-space kernel -(S / 4 pi) dV / r
    const double h = (g.xhi[0] - g.xlo[0]) / g.nx[0];
    for (int d = 0; d < 3; ++d) c->m[d] = 2 * g.nx[d];
    c->MT = (long long)c->m[0] * c->m[1] * c->m[2];
    double2 *h_k = (double2 *)malloc(sizeof(double2) * c->MT);
    if (!h_k) return vp_fail(c, VP_ENOMEM, "host allocation failed");
    const double self = cube_inv_r_mean() / h;
    const double pref = -(g.coupling / (4.0 * M_PI)) * h * h * h;
    for (int a = 0; a < c->m[0]; ++a)
        for (int b = 0; b < c->m[1]; ++b)
            for (int cc = 0; cc < c->m[2]; ++cc) {
                const int ia = a < c->m[0] - a ? a : c->m[0] - a;
                const int ib = b < c->m[1] - b ? b : c->m[1] - b;
                const int ic = cc < c->m[2] - cc ? cc : c->m[2] - cc;
                const double r = h * sqrt((double)ia * ia + (double)ib * ib + (double)ic * ic);
                const double inv = (ia == 0 && ib == 0 && ic == 0) ? self : 1.0 / r;
                h_k[((long long)a * c->m[1] + b) * c->m[2] + cc] = make_double2(pref * inv, 0.0);
            }
    VP_CUDA_TRY(c, cudaMalloc(&c->d_ghat, sizeof(double2) * c->MT));
    VP_CUDA_TRY(c, cudaMalloc(&c->d_fft, sizeof(double2) * c->MT));
    VP_CUDA_TRY(c, cudaMemcpy(c->d_ghat, h_k, sizeof(double2) * c->MT, cudaMemcpyHostToDevice));
    free(h_k);
    VP_CUDA_TRY(c, cudaStreamSynchronize(cudaStreamLegacy));
    for (int d = 2; d >= 0; --d)
        c->launches += fft_launch(c->stream, c->d_ghat, fft_axis(c->m, 3, d, FFT_FWD, c->roots[d], c->sm_count));
    VP_CUDA_TRY(c, cudaGetLastError());
    VP_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    return VP_OK;
}

// ---- launchers ---------------------------------------------------------------

static double cell_volume_v(const vp_grid &g) {
    double dV = 1.0;
    for (int d = 0; d < g.dv; ++d) dV *= (g.vhi[d] - g.vlo[d]) / g.nv[d];
    return dV;
}

template <typename T>
static void moment_launch(vp_ctx *c, double *rho) {
    const T *f = static_cast<const T *>(c->f);
    const double dV = cell_volume_v(c->g);
    if (c->NV <= kWarpCells) {
        // fewer points per block while the grid would leave SMs idle
        const int wpb = c->NX >= 8LL * 2 * c->sm_count ? 8 : 2;
        vp_launch_dep(k_moment<T, true>, nblk(c->NX, wpb), 32 * wpb, 0, c->stream, f, c->NX, c->NV, dV, rho);
    } else {
        vp_launch_dep(k_moment<T, false>, (unsigned)c->NX, kBlock, 0, c->stream, f, c->NX, c->NV, dV, rho);
    }
}

int vp_launch_moment(vp_ctx *c, double *rho) {
    if (c->g.precision == VP_F32) moment_launch<float>(c, rho);
    else moment_launch<double>(c, rho);
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

int vp_launch_poisson(vp_ctx *c, const double *rho, double *phi, double *acc) {
    const vp_grid &g = c->g;
    const int D = g.dx;
    if (c->d_conv) {
        const int n = g.nx[0];
        // every block reads all of rho: outputs that overlap it take a copy
        auto meets = [&](const double *p) { return p && p < rho + n && rho < p + n; };
        if (meets(phi) || meets(acc)) {
            VP_CUDA_TRY(c, cudaMemcpyAsync(c->d_rho, rho, sizeof(double) * n, cudaMemcpyDeviceToDevice, c->stream));
            rho = c->d_rho;
        }
        vp_launch_dep(k_conv1, nblk(n, kConvWarps), 32 * kConvWarps, sizeof(double) * n, c->stream, rho, n,
                      c->d_conv, phi, acc);
        c->launches++;
        VP_CUDA_TRY(c, cudaGetLastError());
        return VP_OK;
    }
    // forward along the last axis (reading rho) .. the second, then the first
    // axis forward, times the Green function, and back; the others back
    for (int d = D - 1; d >= 0; --d) {
        FftLaunch l = fft_axis(c->m, D, d, d ? FFT_FWD : FFT_CONV, c->roots[d], c->sm_count);
        if (d == D - 1) {
            l.f.rho = rho;
            l.f.bg = g.rho_bg;
            for (int k = 0; k < D; ++k) {
                l.f.nbox[k] = g.nx[k];
                l.f.m[k] = c->m[k];
            }
        }
        if (d == 0) {
            l.f.green = c->d_green;
            l.f.ghat = c->d_ghat;
            l.f.scale = 1.0 / (double)c->MT;
        }
        c->launches += fft_launch(c->stream, c->d_fft, l);
    }
    for (int d = 1; d < D; ++d)
        c->launches += fft_launch(c->stream, c->d_fft, fft_axis(c->m, D, d, FFT_INV, c->roots[d], c->sm_count));
    vp_launch_dep(k_force, nblk(c->NX, kBlock), kBlock, 0, c->stream, c->d_fft, phi, acc, force_args(g, c->m,
                  c->NX));
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

template <typename T>
static void diag_part_launch(vp_ctx *c) {
    using W = typename DiagSum<T>::W;
    const vp_grid &g = c->g;
    const int nlast = g.nv[g.dv - 1];
    const long long rows = c->NV / nlast;
    const W *wrow = static_cast<const W *>(c->d_vw);
    const int th = c->NV >= 4096 || nlast > 128 ? 256 : 128;
    vp_launch_dep(k_diag_part<T>, (unsigned)c->NX, th, 0, c->stream, static_cast<const T *>(c->f), c->NV, nlast,
                  make_fastdiv((unsigned)nlast), wrow, wrow + rows, c->vw_unit, cell_volume_v(g), c->d_part,
                  c->d_rho, c->d_flag);
}

// the weights of the kinetic energy, once per context
static int diag_weights(vp_ctx *c) {
    const vp_grid &g = c->g;
    VWeights w{};
    w.dv = g.dv;
    double vmax = 0.0;
    for (int d = 0; d < g.dv; ++d) {
        w.lo[d] = g.vlo[d];
        w.h[d] = (g.vhi[d] - g.vlo[d]) / g.nv[d];
        w.n[d] = g.nv[d];
        vmax = fmax(vmax, fmax(fabs(g.vlo[d]), fabs(g.vhi[d])));
    }
    int e = 0;
    frexp(vmax * vmax, &e);
    w.unit = c->vw_unit = std::isfinite(vmax * vmax) && vmax * vmax > 0.0 ? ldexp(1.0, e) : 1.0;
    const int nlast = g.nv[g.dv - 1];
    const long long rows = c->NV / nlast, most = rows > nlast ? rows : nlast;
    if (g.precision == VP_F32)
        k_vweights<WPair><<<nblk(most, kBlock), kBlock>>>(w, rows, static_cast<WPair *>(c->d_vw),
                                                         static_cast<WPair *>(c->d_vw) + rows);
    else
        k_vweights<double><<<nblk(most, kBlock), kBlock>>>(w, rows, static_cast<double *>(c->d_vw),
                                                          static_cast<double *>(c->d_vw) + rows);
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

int vp_launch_diag(vp_ctx *c, int mode, double *out_dev) {
    const vp_grid &g = c->g;
    // one pass over f gives the density and the velocity sums
    if (g.precision == VP_F32) diag_part_launch<float>(c);
    else diag_part_launch<double>(c);
    c->launches++;
    const int rc = vp_launch_poisson(c, c->d_rho, c->d_phi, c->d_acc);
    if (rc) return rc;
    double dX = 1.0;
    for (int d = 0; d < g.dx; ++d) dX *= (g.xhi[d] - g.xlo[d]) / g.nx[d];
    const long long rest = c->NX / g.nx[0];
    mode %= g.nx[0];
    mode = mode < 0 ? mode + g.nx[0] : mode;
    vp_launch_dep(k_diag_final, nblk(c->NX, kBlock), kBlock, 0, c->stream, c->d_part, c->d_rho, c->d_phi,
                  c->d_acc, c->NX, g.dx, g.nx[0], rest, mode, c->roots[0], c->m[0] / g.nx[0], g.rho_bg, dX,
                  cell_volume_v(g), c->d_diagblk, c->d_diagctr, out_dev);
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

int vp_launch_init_ptr(void *f, const vp_grid &g, int kind, const double *p, int np, cudaStream_t st) {
    IcArgs a{};
    a.kind = kind;
    a.dims = g.dx;
    a.NV = 1;
    long long NX = 1;
    for (int d = 0; d < g.dx; ++d) {
        a.nx[d] = g.nx[d];
        a.nv[d] = g.nv[d];
        a.xlo[d] = g.xlo[d];
        a.vlo[d] = g.vlo[d];
        a.hx[d] = (g.xhi[d] - g.xlo[d]) / g.nx[d];
        a.hv[d] = (g.vhi[d] - g.vlo[d]) / g.nv[d];
        a.xc[d] = 0.5 * (g.xlo[d] + g.xhi[d]);
        a.NV *= g.nv[d];
        NX *= g.nx[d];
    }
    for (int i = 0; i < np && i < 8; ++i) a.p[i] = p[i];
    const long long ncell = NX * a.NV;
    if (g.precision == VP_F32)
        k_init<float><<<nblk(ncell, kBlock), kBlock, 0, st>>>(static_cast<float *>(f), ncell, a);
    else
        k_init<double><<<nblk(ncell, kBlock), kBlock, 0, st>>>(static_cast<double *>(f), ncell, a);
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

int vp_launch_init(vp_ctx *c, int kind, const double *p, int np) {
    const int rc = vp_launch_init_ptr(c->f, c->g, kind, p, np, c->stream);
    c->launches++;
    if (rc) return vp_fail(c, rc, "initial condition launch failed");
    return VP_OK;
}

// ---- allocation-free periodic Poisson solve ------------------------------------
// vp_poisson_periodic_noalloc: the periodic solve of vp_poisson_solve for
// callers that must not allocate device memory.  Its complex FFT work array is
// this file-scope device array (VP_NOALLOC_MAX_POINTS complex doubles, 4 MiB,
// held by every device that loads the library until the process exits); the
// Green function is evaluated on the fly instead of read from a table.  The
// array is shared by all calls: calls that overlap on the GPU race on it.

static __device__ __align__(256) double2 g_noalloc_fft[VP_NOALLOC_MAX_POINTS];

namespace {

constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mu;
double2 *g_noalloc_dev_ptr[kNoallocMaxDevices];
int g_noalloc_sms[kNoallocMaxDevices];

__device__ double noalloc_stencil_eig(int order, double theta) {
    // eigenvalue of the symmetric discrete Laplacian stencil (b_0..b_3)/den
    // (Eqs. C1, C5, C6) times h^2: -(4/den) sum_m b_m sin^2(m theta / 2)
    double b1 = 1.0, b2 = 0.0, b3 = 0.0, den = 1.0;
    if (order == 4) {
        b1 = 16.0;
        b2 = -1.0;
        den = 12.0;
    } else if (order == 6) {
        b1 = 270.0;
        b2 = -27.0;
        b3 = 2.0;
        den = 180.0;
    }
    const double s1 = sin(0.5 * theta), s2 = sin(theta), s3 = sin(1.5 * theta);
    return -4.0 * (b1 * s1 * s1 + b2 * s2 * s2 + b3 * s3 * s3) / den;
}

// multiply every Fourier mode by S / lambda(k) / NX (k = 0 -> 0)
__global__ void k_green_onfly(double2 *__restrict__ a, long long NX, int dims, int3 n, double3 h,
                              int order, double S) {
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= NX) return;
    const int nn[3] = {n.x, n.y, n.z};
    const double hh[3] = {h.x, h.y, h.z};
    long long r = x;
    bool allzero = true;
    double lam = 0.0;
    for (int d = dims - 1; d >= 0; --d) {
        const long long k = r % nn[d];
        r /= nn[d];
        if (k) allzero = false;
        lam += noalloc_stencil_eig(order, 2.0 * 3.141592653589793238462643383279502884 * (double)k / (double)nn[d]) /
               (hh[d] * hh[d]);
    }
    const double sc = allzero ? 0.0 : S / lam / (double)NX;
    a[x] = make_double2(a[x].x * sc, a[x].y * sc);
}

}  // namespace

extern "C" int vp_poisson_periodic_noalloc(const vp_grid *g, void *cuda_stream, const double *rho_dev,
                                           double *phi_dev, double *accel_dev) {
    if (!g || !rho_dev || !accel_dev) return VP_EINVAL;
    if (g->dx < 1 || g->dx > 3 || g->poisson != VP_POIS_PERIODIC) return VP_EINVAL;
    if (g->pois_order != 2 && g->pois_order != 4 && g->pois_order != 6) return VP_EINVAL;
    if (!std::isfinite(g->coupling) || !std::isfinite(g->rho_bg)) return VP_EINVAL;
    const int D = g->dx;
    long long NX = 1;
    for (int d = 0; d < D; ++d) {
        if (g->nx[d] < 1 || g->nx[d] > 4096) return VP_EINVAL;
        if (!(g->xhi[d] > g->xlo[d]) || !std::isfinite(g->xhi[d]) || !std::isfinite(g->xlo[d]))
            return VP_EINVAL;
        NX *= g->nx[d];
    }
    if (NX > VP_NOALLOC_MAX_POINTS) return VP_EINVAL;
    // an error left by earlier work would be indistinguishable from ours at
    // the end: report it (and leave it pending) before launching anything
    if (cudaPeekAtLastError() != cudaSuccess) return VP_ECUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return VP_ECUDA;
    double2 *buf = nullptr;
    int sms = 0;
    {
        // once per device, with that device current: the device address of the
        // static array (its name in host code is only a host-side stand-in)
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_dev_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_fft) != cudaSuccess || !p) return VP_ECUDA;
            if (cudaFuncSetAttribute(k_fft_lines, cudaFuncAttributeMaxDynamicSharedMemorySize, kFftSmem) !=
                    cudaSuccess ||
                cudaDeviceGetAttribute(&g_noalloc_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
                return VP_ECUDA;
            g_noalloc_dev_ptr[dev] = static_cast<double2 *>(p);
        }
        buf = g_noalloc_dev_ptr[dev];
        sms = g_noalloc_sms[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int3 nb = make_int3(g->nx[0], D > 1 ? g->nx[1] : 1, D > 2 ? g->nx[2] : 1);
    const int m[3] = {nb.x, nb.y, nb.z};
    // every element of the work array that is read is written first: no clearing needed
    for (int d = D - 1; d >= 0; --d) {
        FftLaunch l = fft_axis(m, D, d, FFT_FWD, nullptr, sms);
        if (d == D - 1) {
            l.f.rho = rho_dev;
            l.f.bg = g->rho_bg;
            for (int k = 0; k < D; ++k) l.f.nbox[k] = l.f.m[k] = m[k];
        }
        fft_launch(st, buf, l);
    }
    const double3 h = make_double3((g->xhi[0] - g->xlo[0]) / g->nx[0],
                                   D > 1 ? (g->xhi[1] - g->xlo[1]) / g->nx[1] : 1.0,
                                   D > 2 ? (g->xhi[2] - g->xlo[2]) / g->nx[2] : 1.0);
    k_green_onfly<<<nblk(NX, kBlock), kBlock, 0, st>>>(buf, NX, D, nb, h, g->pois_order, g->coupling);
    for (int d = 0; d < D; ++d) fft_launch(st, buf, fft_axis(m, D, d, FFT_INV, nullptr, sms));
    vp_launch_dep(k_force, nblk(NX, kBlock), kBlock, 0, st, buf, phi_dev, accel_dev, force_args(*g, m, NX));
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

// vp_fluxnet.cu -- learned flux correction on a coarser velocity grid
// (an addition to the method, not in the paper).
//
// A 25 -> 32 -> 32 -> 32 -> 1 ReLU network g corrects the mass that a
// coarse-grid spatial sweep moves through an interface:
//   M = nu Phi_MP + s g(x),
// Phi_MP the CSL7 flux after the MP constraint, s = max |u| over the 8-cell
// upwind-ordered stencil u_{-3..4}, x = ((u_k - u_0) / s, (u+_k - u-_k) / (2 s),
// (u+_k + u-_k - 2 u_k) / (2 s), nu) with u+ / u- the same cells of the lines in
// the neighbouring velocity cells (+: larger |v|).  The correction is a mass, not a flux value: the
// sub-cell spread of speeds inside a coarse velocity cell moves mass even
// where the cell's own fractional shift nu is small.  The corrected mass
// passes the PP limiter (f_i - 2 M >= 0, f_{i+1} + 2 M >= 0) and, on request
// (use_net = 2), the MP bounds of App. A before it (the clamp into
// [nu f_min, nu f_max]); the update keeps the flux form
// f'_i = f_{i-n} - (M_out - M_in), so conservation and f >= 0 hold exactly as
// for the plain scheme.  Weights and matrix inputs are bfloat16, sums FP32.
//
// Training data come from fine-grid runs of the method itself: for a sweep,
// the fine-grid mass through every coarse interface (mean over the fine
// lines a coarse line aggregates), minus the coarse integer-shift part and
// the coarse MP-limited fractional mass, over s, is the target of g.
// Training: forward and backward on the tensor cores, a tile of 16 samples per
// warp (bfloat16-rounded weights, inputs and activations, FP32 sums, deltas in
// three bfloat16 terms, straight-through backward), weight gradients summed per
// CTA, Adam.
#include <cuda_bf16.h>

#include <atomic>
#include <cmath>

#include "vp_internal.cuh"
#include "vp_sum.cuh"
#include "vp_sweep_core.cuh"
#include "vp_umma.cuh"

namespace {

using vp_sum::PairSum;
using vp_sum::widen;

constexpr int H = VP_NET_HIDDEN;
constexpr int NF = VP_NET_FEATURES;

// parameter layout (floats): W1[H][NF] b1[H] W2[H][H] b2[H] W3[H][H] b3[H] w4[H] b4[1]
constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + H * NF;
constexpr int OFF_W2 = OFF_B1 + H;
constexpr int OFF_B2 = OFF_W2 + H * H;
constexpr int OFF_W3 = OFF_B2 + H;
constexpr int OFF_B3 = OFF_W3 + H * H;
constexpr int OFF_W4 = OFF_B3 + H;
constexpr int OFF_B4 = OFF_W4 + H;
constexpr int NPARAM = OFF_B4 + 1;
static_assert(NPARAM == VP_NET_NPARAM, "parameter count");

__device__ __forceinline__ float bfr(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// features of the upwind-ordered stencil u[0..7] = u_{-3..4} and of the same
// cells up / um of the velocity-neighbour lines (+: larger |v|): velocity
// difference and curvature
__device__ __forceinline__ float net_features(const float *u, const float *up, const float *um, float nu,
                                              float *x) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s = fmaxf(s, fabsf(u[k]));
    s += 1e-30f;
    const float inv = 1.0f / s;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = (u[k] - u[3]) * inv;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[8 + k] = (up[k] - um[k]) * (0.5f * inv);
#pragma unroll
    for (int k = 0; k < 8; ++k) x[16 + k] = fmaf(0.5f, up[k] + um[k], -u[k]) * inv;
    x[24] = nu;
    return s;
}

// ---- training ----------------------------------------------------------------------

// Loss and gradient on the tensor cores.  A warp takes tiles of 16 samples and
// keeps a tile's whole forward and backward pass in registers: the accumulators
// of mma.sync m16n8k16 are, packed to bfloat16, the A operand of the next layer,
// and an 8x8 transpose of such a register (movmatrix) is the operand of the
// weight gradients, whose contraction runs over the samples.  (tcgen05 needs
// 128-row operands in shared memory and a barrier round trip per layer; three
// chained 32 x 32 layers of 16 rows are all latency there.)
//   forward   Z = W A + b: bfloat16 operands as defined, FP32 sums, and those
//             whose last bits could decide the bfloat16 activation once more,
//             exactly (activate);
//   backward  the FP32 deltas are split into three bfloat16 terms (24 bits), so
//             that no bit of them is lost: dA = W^T delta, dW += delta A^T.
// Weight gradients stay in registers over all of a warp's tiles, are summed over
// the CTA in shared memory and added to global memory once per CTA.
// A training step of 32 768 samples: 65 -> 27.3 us; with one thread per sample and
// both operands of every FMA read from shared memory the LSU pipe set the time
// (67% busy, 256 CTAs of 75 KB, 10% of the warps).
// Samples come in consecutive groups of `group` (1 or 2; a pair = the two
// interfaces of one cell) whose residual is r = sum_k a_k (g_k - y_k) (a_k =
// coef[k], 1 without coef); the loss is the mean of r^2 over groups.
constexpr int kTrainWarps = 8;
constexpr int kTrainThreads = 32 * kTrainWarps;

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ uint32_t transpose8x8(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
// bf16(lo) in the low half, bf16(hi) in the high half
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}
// bf16(max(lo, 0)) in the low half, bf16(max(hi, 0)) in the high half
__device__ __forceinline__ uint32_t pack_relu_bf16(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}
__device__ __forceinline__ float low_half(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float high_half(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }

// A matrix of 16 rows (samples) x 32 columns as packed 8x8 blocks: m[h][c] holds
// rows 8h + lane / 4, columns 8c + 2 (lane % 4) and the next
struct Tile16 {
    uint32_t m[2][4];
    // A operand of the k-step j (columns 16j .. 16j + 15)
    __device__ __forceinline__ void operand(int j, uint32_t (&a)[4]) const {
        a[0] = m[0][2 * j];
        a[1] = m[1][2 * j];
        a[2] = m[0][2 * j + 1];
        a[3] = m[1][2 * j + 1];
    }
    __device__ __forceinline__ Tile16 transposed() const {
        Tile16 t;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int c = 0; c < 4; ++c) t.m[h][c] = transpose8x8(m[h][c]);
        return t;
    }
};

// acc[c] += A B for the four 8-column blocks c of B, whose operands lie in shared
// memory in lane order: ops[(4 j + c) 32 + lane]
__device__ __forceinline__ void times(float (&acc)[4][4], const Tile16 &A, const uint2 *ops, int lane) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        uint32_t a[4];
        A.operand(j, a);
#pragma unroll
        for (int c = 0; c < 4; ++c) mma16816(acc[c], a, ops[(4 * j + c) * 32 + lane]);
    }
}

// one of the three bfloat16 terms of d (what is left of it stays in d)
__device__ __forceinline__ Tile16 take_term(float (&d)[4][4]) {
    Tile16 t;
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t p = pack2(d[c][2 * h], d[c][2 * h + 1]);
            t.m[h][c] = p;
            d[c][2 * h] -= low_half(p);
            d[c][2 * h + 1] -= high_half(p);
        }
    return t;
}

// dW (32 outputs x 32 inputs, in 16 x 8 blocks) += delta^T A, over the 16 samples
__device__ __forceinline__ void outer(float (&dw)[2][4][4], const Tile16 &dt, const Tile16 &at) {
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const uint32_t a[4] = {dt.m[0][2 * m], dt.m[0][2 * m + 1], dt.m[1][2 * m], dt.m[1][2 * m + 1]};
#pragma unroll
        for (int c = 0; c < 4; ++c) mma16816(dw[m][c], a, make_uint2(at.m[0][c], at.m[1][c]));
    }
}

// one layer of the backward pass: d = delta of the layer (destroyed); dw, db of
// the layer; with ops (the layer's W^T) da = W^T delta
template <bool DGRAD>
__device__ __forceinline__ void backward(float (&d)[4][4], const Tile16 &in, const uint2 *ops, int lane,
                                         float (&dw)[2][4][4], float (&db)[4][2], float (&da)[4][4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        db[c][0] += d[c][0] + d[c][2];
        db[c][1] += d[c][1] + d[c][3];
#pragma unroll
        for (int k = 0; k < 4; ++k) da[c][k] = 0.f;
    }
    const Tile16 at = in.transposed();
    const Tile16 t0 = take_term(d), t1 = take_term(d), t2 = take_term(d);
    // smallest terms first
#pragma unroll
    for (int k = 2; k >= 0; --k) {
        const Tile16 &t = k == 0 ? t0 : (k == 1 ? t1 : t2);
        outer(dw, t.transposed(), at);
        if (DGRAD) times(da, t, ops, lane);
    }
}

// The sum z of row `row`, column `col` of a layer in fixed point, a product per
// lane: 44 bits below the largest possible product `most`, rounded once to FP32.
__device__ __forceinline__ float exact_sum(const Tile16 &in, const uint2 *ops, float bias, int row, int col, float most,
                                           int lane) {
    // lane k: input k of the row, weight k of the column
    uint32_t ap = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t v = __shfl_sync(0xffffffffu, row & 8 ? in.m[1][c] : in.m[0][c], 4 * (row & 7) + ((lane >> 1) & 3));
        if (lane >> 3 == c) ap = v;
    }
    const uint2 wp = ops[(4 * (lane >> 4) + (col >> 3)) * 32 + 4 * (col & 7) + ((lane >> 1) & 3)];
    const uint32_t w = lane & 8 ? wp.y : wp.x;
    const float prod = lane & 1 ? high_half(ap) * high_half(w) : low_half(ap) * low_half(w);  // exact
    // units of 2^(e - 22), then of 2^(e - 44), 2^e > most
    const int e = (int)(__float_as_uint(most) >> 23) - 126;
    const float up = __uint_as_float((unsigned)(127 + 22 - e) << 23), q = prod * up, hi = rintf(q);
    const int sh = __reduce_add_sync(0xffffffffu, (int)hi);
    const int sl = __reduce_add_sync(0xffffffffu, __float2int_rn((q - hi) * 4194304.f));
    const float bq = bias * up, bh = rintf(bq);
    const long long sum = ((long long)sh << 22) + sl + (((long long)bh << 22) + __float2int_rn((bq - bh) * 4194304.f));
    return __fmul_rn(__ll2float_rn(sum), __uint_as_float((unsigned)(127 - 44 + e) << 23));
}

// relu(z) rounded to bfloat16, z = W in + bias the layer's FP32 sums.  Where their
// error could carry a sum over a rounding boundary or over zero, the activation
// moves by 2^-9 of itself (or a gradient appears), and the loss adds such moves up:
// single sums decide the sixth digit of a batch's loss.  So sums whose activation
// changes within +- tau are done again exactly, about two of a tile's 1536.
// tau = kSettle (max |in| reach.x + reach.y), reach = {largest sum |w| of a column,
// largest |b|}: the tensor cores' accumulators stay well inside for sums whose terms
// cancel (2^-26 suffices) and inside where they all add up (2^-25 misses a few).
// Error of the loss and of the gradient against 64-bit sums, rms of 12 batches of
// 4000, 32 768 and 600 000 samples: 1.9e-7, 2.1e-7, 2.0e-7 and 1.8e-7, 1.7e-7,
// 2.4e-7; without 2.6e-6, 5.9e-7, 3.5e-7 and 8.9e-6, 2.9e-6, 1.6e-6; with chains of
// FP32 FMAs for all sums 1.3e-6, 4.2e-7, 2.3e-7 and 7.0e-6, 3.0e-6, 1.4e-6.  It
// takes 2.5 of a training step's 27.3 us (the FMA chains: 2.0).
constexpr float kSettle = 0x1p-24f;
__device__ __forceinline__ Tile16 activate(const float (&z)[4][4], const Tile16 &in, const uint2 *ops,
                                           const float2 *bias, float2 reach, int lane) {
    Tile16 t;
    float amax[2], tau[2];
    uint32_t any = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        auto mag = [&](uint32_t p) {
            p &= 0x7fff7fffu;
            return *reinterpret_cast<const __nv_bfloat162 *>(&p);
        };
        __nv_bfloat162 m = __hmax2(__hmax2(mag(in.m[h][0]), mag(in.m[h][1])), __hmax2(mag(in.m[h][2]), mag(in.m[h][3])));
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) m = __hmax2(m, __shfl_xor_sync(0xffffffffu, m, o));
        amax[h] = fmaxf(__low2float(m), __high2float(m));
        const float v = fmaf(amax[h], reach.x, reach.y);
        tau[h] = amax[h] > 0.f && v > 1e-20f && v < 1e20f ? v * kSettle : 0.f;  // no inputs: z = b, exact
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float u = fmaxf(z[c][2 * h], -tau[h]), v = fmaxf(z[c][2 * h + 1], -tau[h]);
            t.m[h][c] = pack_relu_bf16(u - tau[h], v - tau[h]);
            any |= t.m[h][c] ^ pack_relu_bf16(u + tau[h], v + tau[h]);
        }
    }
    uint32_t who = __ballot_sync(0xffffffffu, any != 0);
    if (who == 0) return t;
    uint32_t mine = 0;  // bit 8 h + 2 c + i: row 8 h + lane / 4, column 8 c + 2 (lane % 4) + i
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float u = fmaxf(z[c][2 * h], -tau[h]), v = fmaxf(z[c][2 * h + 1], -tau[h]);
            const uint32_t d = t.m[h][c] ^ pack_relu_bf16(u + tau[h], v + tau[h]);
            mine |= (d & 0xffffu ? 1u : 0u) << (8 * h + 2 * c) | (d >> 16 ? 2u : 0u) << (8 * h + 2 * c);
        }
    while (who) {
        const int src = __ffs(who) - 1;
        const uint32_t his = __shfl_sync(0xffffffffu, mine, src);
        const int j = __ffs(his) - 1;
        const int row = (src >> 2) + (j & 8), col = (j & 6) * 4 + 2 * (src & 3) + (j & 1);
        const float most = __shfl_sync(0xffffffffu, j & 8 ? amax[1] : amax[0], src) * reach.x;
        const float v = exact_sum(in, ops, reinterpret_cast<const float *>(bias)[col], row, col,
                                  fmaxf(most, reach.y), lane);
        if (lane == src) {
            const uint32_t p = pack2(fmaxf(v, 0.f), fmaxf(v, 0.f)), keep = j & 1 ? 0x0000ffffu : 0xffff0000u;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i == j >> 1) t.m[i >> 2][i & 3] = (t.m[i >> 2][i & 3] & keep) | (p & ~keep);
            mine &= mine - 1;
        }
        if ((his & (his - 1)) == 0) who &= who - 1;
    }
    return t;
}
// d where the activation is positive, 0 elsewhere
__device__ __forceinline__ void mask(float (&d)[4][4], const Tile16 &t) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (!(t.m[h][c] & 0x7fffu)) d[c][2 * h] = 0.f;
            if (!(t.m[h][c] & 0x7fff0000u)) d[c][2 * h + 1] = 0.f;
        }
}

constexpr int kTrainOps = 8 * 32;  // operands (uint2) of one 32 x 32 layer
constexpr size_t kTrainSmem = (size_t)5 * kTrainOps * sizeof(uint2) + (size_t)kTrainWarps * NPARAM * sizeof(float) + 16;

__global__ void __launch_bounds__(kTrainThreads, 1) k_net_grad(const float *__restrict__ X,
                                                               const float *__restrict__ y,
                                                               const float *__restrict__ coef,
                                                               const float *__restrict__ wts, long long nsamp,
                                                               int group, float *__restrict__ grad,
                                                               float *__restrict__ loss) {
    extern __shared__ __align__(16) unsigned char gsm[];
    uint2 *ops = reinterpret_cast<uint2 *>(gsm);  // W1 W2 W3, then W2^T W3^T
    float *sums = reinterpret_cast<float *>(ops + 5 * kTrainOps);  // [warp][NPARAM]
    __shared__ float sloss[kTrainWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t2 = 2 * (lane & 3);
    // B operand of W (n = output, k = input): rows k = 16 j + t2 (+1, +8, +9),
    // column n = 8 c + g; of W^T the roles of k and n swapped
    for (int e = threadIdx.x; e < 5 * kTrainOps; e += blockDim.x) {
        const int m = e / kTrainOps, l = e & 31, c = (e >> 5) & 3, j = (e >> 7) & 1;
        const int n = 8 * c + (l >> 2), k = 16 * j + 2 * (l & 3);
        auto w = [&](int kk) -> float {
            if (m == 0) return kk < NF ? wts[OFF_W1 + n * NF + kk] : 0.f;
            if (m == 1) return wts[OFF_W2 + n * H + kk];
            if (m == 2) return wts[OFF_W3 + n * H + kk];
            return wts[(m == 3 ? OFF_W2 : OFF_W3) + kk * H + n];
        };
        ops[e] = make_uint2(pack2(w(k), w(k + 1)), pack2(w(k + 8), w(k + 9)));
    }
    __shared__ float2 vecs[4][16];  // b1 b2 b3 w4, two columns each
    if (threadIdx.x < 128) {
        const int v = threadIdx.x >> 5, col = threadIdx.x & 31;
        const float w = wts[(v == 0 ? OFF_B1 : (v == 1 ? OFF_B2 : (v == 2 ? OFF_B3 : OFF_W4))) + col];
        reinterpret_cast<float *>(vecs[v])[col] = v == 3 ? bfr(w) : w;
    }
    const float b4 = wts[OFF_B4];
    __shared__ float2 reach[3];
    __syncthreads();
    if (threadIdx.x < 96) {
        const int m = threadIdx.x >> 5, n = threadIdx.x & 31;
        float a = 0.f, b = fabsf(reinterpret_cast<const float *>(vecs[m])[n]);
        for (int e = 0; e < 8; ++e) {
            const uint2 w = ops[m * kTrainOps + (4 * (e >> 2) + (n >> 3)) * 32 + 4 * (n & 7) + (e & 3)];
            a += (fabsf(low_half(w.x)) + fabsf(high_half(w.x))) + (fabsf(low_half(w.y)) + fabsf(high_half(w.y)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
            b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
        }
        if (n == 0) reach[m] = make_float2(a, b);
    }
    __syncthreads();
    float dw1[2][4][4] = {}, dw2[2][4][4] = {}, dw3[2][4][4] = {};
    float db1[4][2] = {}, db2[4][2] = {}, db3[4][2] = {}, dw4[4][2] = {};
    float db4 = 0.f, lsum = 0.f;
    const float ngroups = (float)(nsamp / group);
    const long long ntiles = (nsamp + 15) / 16;
    // tiles over the CTAs first, so that few of them still use every SM
    for (long long tile = blockIdx.x + (long long)warp * gridDim.x; tile < ntiles;
         tile += (long long)kTrainWarps * gridDim.x) {
        const long long s0 = tile * 16 + g;
        const bool ok[2] = {s0 < nsamp, s0 + 8 < nsamp};
        Tile16 x;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int col = 8 * c + t2;
                const float *p = X + (s0 + 8 * h) * NF + col;
                const float lo = ok[h] && col < NF ? __ldg(p) : 0.f, hi = ok[h] && col + 1 < NF ? __ldg(p + 1) : 0.f;
                x.m[h][c] = pack2(lo, hi);
            }
        float yv[2], av[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            yv[h] = ok[h] ? __ldg(y + s0 + 8 * h) : 0.f;
            av[h] = ok[h] ? (coef ? __ldg(coef + s0 + 8 * h) : 1.f) : 0.f;
        }
        float z[4][4];
        auto start = [&](int v) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 b = vecs[v][4 * c + (lane & 3)];
                z[c][0] = z[c][2] = b.x;
                z[c][1] = z[c][3] = b.y;
            }
        };
        start(0);
        times(z, x, ops, lane);
        const Tile16 h1 = activate(z, x, ops, vecs[0], reach[0], lane);
        start(1);
        times(z, h1, ops + kTrainOps, lane);
        const Tile16 h2 = activate(z, h1, ops + kTrainOps, vecs[1], reach[1], lane);
        start(2);
        times(z, h2, ops + 2 * kTrainOps, lane);
        const Tile16 h3 = activate(z, h2, ops + 2 * kTrainOps, vecs[2], reach[2], lane);
        // the output, the residual and the delta of the output
        float dg[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float o = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 w4 = vecs[3][4 * c + (lane & 3)];
                o = fmaf(w4.x, low_half(h3.m[h][c]), o);
                o = fmaf(w4.y, high_half(h3.m[h][c]), o);
            }
            o += __shfl_xor_sync(0xffffffffu, o, 1);
            o += __shfl_xor_sync(0xffffffffu, o, 2);
            const float term = ok[h] ? av[h] * ((o + b4) - yv[h]) : 0.f;
            float r = term;
            if (group == 2) r += __shfl_xor_sync(0xffffffffu, term, 4);  // the pair's other row
            dg[h] = ok[h] ? 2.0f * r * av[h] / ngroups : 0.f;
            if (t2 == 0) {
                db4 += dg[h];
                if (ok[h] && (group == 1 || (g & 1) == 0)) lsum += r * r / ngroups;
            }
        }
        float d[4][4], da[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                dw4[c][0] = fmaf(dg[h], low_half(h3.m[h][c]), dw4[c][0]);
                dw4[c][1] = fmaf(dg[h], high_half(h3.m[h][c]), dw4[c][1]);
                const float2 w4 = vecs[3][4 * c + (lane & 3)];
                d[c][2 * h] = dg[h] * w4.x;
                d[c][2 * h + 1] = dg[h] * w4.y;
            }
        mask(d, h3);
        backward<true>(d, h2, ops + 4 * kTrainOps, lane, dw3, db3, da);
        mask(da, h2);
        backward<true>(da, h1, ops + 3 * kTrainOps, lane, dw2, db2, d);
        mask(d, h1);
        backward<false>(d, x, nullptr, lane, dw1, db1, da);
    }
    // the warp's sums to shared memory, in the parameters' order
    float *q = sums + warp * NPARAM;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int row = 16 * m + g + 8 * (k >> 1), col = 8 * c + t2 + (k & 1);
                if (col < NF) q[OFF_W1 + row * NF + col] = dw1[m][c][k];
                q[OFF_W2 + row * H + col] = dw2[m][c][k];
                q[OFF_W3 + row * H + col] = dw3[m][c][k];
            }
    auto over_rows = [&](float v) -> float {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float s1 = over_rows(db1[c][i]), s2 = over_rows(db2[c][i]), s3 = over_rows(db3[c][i]),
                        s4 = over_rows(dw4[c][i]);
            if (g == 0) {
                const int col = 8 * c + t2 + i;
                q[OFF_B1 + col] = s1;
                q[OFF_B2 + col] = s2;
                q[OFF_B3 + col] = s3;
                q[OFF_W4 + col] = s4;
            }
        }
    db4 = over_rows(db4);
    lsum = over_rows(lsum);
    if (lane == 0) {
        q[OFF_B4] = db4;
        sloss[warp] = lsum;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kTrainWarps; ++k) v += sums[k * NPARAM + i];
        atomicAdd(grad + i, v);
    }
    if (threadIdx.x == 0) {
        float v = 0.f;
        for (int k = 0; k < kTrainWarps; ++k) v += sloss[k];
        atomicAdd(loss, v);
    }
}

__global__ void k_adam(float *__restrict__ wts, float *__restrict__ m, float *__restrict__ v,
                       float *__restrict__ grad, int n, float lr, float b1, float b2, float eps, float bc1,
                       float bc2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = grad[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    wts[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    grad[i] = 0.f;
}

// ---- training data -----------------------------------------------------------------

// FP64 instructions take 16 cycles each here, conversions included, and the
// outputs are tens of millions of doubles: sums of a few floats are kept as a
// value and its error term (vp_sum.cuh).
__device__ __forceinline__ double pair_value(const PairSum &p) { return widen(p.s) + widen(p.e); }

// geometry of the line kernels below: lines of L cells at stride inner, W (a
// power of two, at most kTileLines) consecutive lines per CTA
constexpr int kTileLines = 64;

struct LineTile : LineShape {
    int W, logW;
};
// element of a line's first cell, and its class
struct LinePos {
    long long base[kTileLines];
    unsigned cls[kTileLines];
};
__device__ __forceinline__ void place_lines(const LineTile &q, long long l0, int nl, LinePos &p) {
    for (int i = threadIdx.x; i < nl; i += blockDim.x) p.cls[i] = q.place(l0 + i, p.base[i]);
}

// rows beyond the line that the 7- and 8-cell stencils reach (zero, or the
// wrapped cells of a periodic line)
constexpr int kEdge = 8;

__device__ __forceinline__ int wrap_row(int r, int L) {
    while (r < 0) r += L;
    while (r >= L) r -= L;
    return r;
}

// Stage nl lines (base elements plus `off`; a line with use(i) false is zero):
// at(line, row) is the place of rows -kEdge .. L + kEdge - 1.  Lanes run over
// the lines where neighbouring lines are neighbours in memory, else along the
// line; every cell's copy is in flight at once (vp_tma::cp_async_wait_all and a
// barrier complete them).
template <typename Use, typename At>
__device__ __forceinline__ void stage_lines(const float *__restrict__ f, const LineTile &q, const LinePos &p, int nl,
                                            long long off, Use use, At at) {
    const int R = q.L + 2 * kEdge;
    auto cell = [&](const float *line, bool in, float *to, int row) {
        int r = row;
        if (q.periodic) r = wrap_row(r, q.L);
        else in = in && r >= 0 && r < q.L;
        if (in) vp_tma::cp_async<4>(to, line + (long long)r * q.inner);
        else *to = 0.f;
    };
    if (q.inner >= 16) {
        const int i = threadIdx.x & (q.W - 1);
        if (i >= nl) return;
        const bool in = use(i);
        const float *line = f + p.base[i] + off;
        for (int row = (int)(threadIdx.x >> q.logW) - kEdge; row < q.L + kEdge; row += blockDim.x >> q.logW)
            cell(line, in, at(i, row), row);
    } else {
        for (int i = threadIdx.x >> 5; i < nl; i += blockDim.x >> 5) {
            const bool in = use(i);
            for (int r = (threadIdx.x & 31); r < R; r += 32) cell(f + p.base[i] + off, in, at(i, r - kEdge), r - kEdge);
        }
    }
}

// The same for lines that lie side by side in fours on 16-byte boundaries
// (rows of `pitch` floats, a multiple of four, from row -kEdge at u): 16-byte
// copies.  4-byte ones are as many copy instructions as cells, whose rate, and
// not HBM's, set the time (training samples of a 64 x 128 per axis 2D2V grid,
// of which these lines are half: 1065 -> 932 us).
__device__ __forceinline__ void stage_quads(const float *__restrict__ f, const LineTile &q, const LinePos &p, int nl,
                                            float *u, int pitch) {
    const int i = 4 * (int)(threadIdx.x & ((q.W >> 2) - 1));
    if (i >= nl) return;
    const float *line = f + p.base[i];
    for (int row = (int)(threadIdx.x >> (q.logW - 2)) - kEdge; row < q.L + kEdge; row += blockDim.x >> (q.logW - 2)) {
        float *to = u + row * pitch + i;
        const int r = q.periodic ? wrap_row(row, q.L) : row;
        if (r >= 0 && r < q.L)
            vp_tma::cp_async16(to, line + (long long)r * q.inner);
        else
            *reinterpret_cast<float4 *>(to) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Mass through interfaces of fine lines, in fine-cell units, for one sweep:
// G_{i+1/2} = sum of the N whole cells swept through + nu Phi_hat at the
// shifted interface (the flux form of the SL update: f'_i = f_i + G_{i-1/2}
// - G_{i+1/2}).  Output: G[line][j] at interfaces j * every - 1/2 for j = 0 ..
// L/every (boundary interfaces included).
// A CTA stages W lines and the block of results, which it writes as one
// contiguous run (one thread per line, its results in rows of its own, its
// stencil from global memory and double-precision prefix sums took 2783 us for
// 6.7e7 cells; the output alone is 80 us of HBM; now ~400 us, bound by issue).  Whole-cell parts of at most
// kFewCells cells are summed directly; PREFIX: longer ones from double prefix
// sums of the line.
constexpr int kFewCells = 8;

template <bool PREFIX, bool QUAD>
__global__ void __launch_bounds__(256) k_fine_flux(const float *__restrict__ f, LineTile q,
                                                   const LineShift<float> *__restrict__ tab, int every,
                                                   double *__restrict__ G, float alpha) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int L = q.L, W = q.W, nout = L / every + 1, NP = nout | 1, WP = QUAD ? W : W + 1;
    double *Gs = reinterpret_cast<double *>(fsm);            // [W][NP]
    double *S = Gs + W * NP;                                  // PREFIX: [L + 1][W]
    float *u = reinterpret_cast<float *>(S + (PREFIX ? (L + 1) * W : 0)) + kEdge * WP;  // rows of WP, from row -kEdge
    __shared__ LinePos pos;
    const long long l0 = (long long)blockIdx.x * W;
    const int nl = (int)(q.lines - l0 < W ? q.lines - l0 : W);
    place_lines(q, l0, nl, pos);
    __syncthreads();
    if (QUAD)
        stage_quads(f, q, pos, nl, u, WP);
    else
        stage_lines(f, q, pos, nl, 0, [](int) { return true; }, [&](int i, int row) { return u + row * WP + i; });
    vp_tma::cp_async_wait_all();
    __syncthreads();
    if (PREFIX) {
        for (int i = threadIdx.x; i < nl; i += blockDim.x) {
            double a = 0.0;
            for (int k = 0; k < L; ++k) {
                S[k * W + i] = a;
                a += widen(u[k * WP + i]);
            }
            S[L * W + i] = a;
        }
        __syncthreads();
    }
    const int i = threadIdx.x & (W - 1);
    if (i < nl) {
        const LineShift<float> sh = tab[pos.cls[i]];
        const int sg = sh.sigma;
        const int n = sh.n * sg;  // whole cells swept, in the upwind frame
        // the shift of the stencil: modulo the line, or just off its ends
        const int ns = q.periodic ? n % L : (n < -2 * L - 8 ? -2 * L - 8 : (n > 2 * L + 8 ? 2 * L + 8 : n));
        const float *ui = u + i;
        bool over = false;  // a pair sum left the float range (or a cell is not finite)
        // the mass through interface j, M the fractional one in the upwind frame
        auto emit = [&](int j, float M) {
            const int c = j * every;
            double g;
            if (PREFIX) {
                // sum of the cells before k, extended beyond the line
                auto upto = [&](int k) -> double {
                    if (q.periodic) {
                        int w0 = k / L, r = k - w0 * L;
                        if (r < 0) {
                            r += L;
                            --w0;
                        }
                        return S[r * W + i] + (double)w0 * S[L * W + i];
                    }
                    return S[(k < 0 ? 0 : (k > L ? L : k)) * W + i];
                };
                // cells c - n .. c - 1 (swept rightwards) or c .. c + n - 1
                g = (sg > 0 ? upto(c) - upto(c - n) : upto(c + n) - upto(c)) + widen(M);
                g = sg > 0 ? g : -g;
            } else {
                // |n| < kFewCells: the cells lie within the staged rows
                if (n == 0) {
                    M = __fadd_rn(M, 0.f);  // (the sum of no cells and M: no -0)
                    Gs[i * NP + j] = widen(sg > 0 ? M : -M);
                    return;
                }
                PairSum p;
                const float *v = ui + (sg > 0 ? (n >= 0 ? c - n : c) : (n >= 0 ? c : c + n)) * WP;
                const float one = n >= 0 ? 1.f : -1.f;
                for (int m = n >= 0 ? n : -n; m > 0; --m, v += WP) p.add(one * *v);
                p.add(M);
                over |= !isfinite(p.s);
                p.s = sg > 0 ? p.s : -p.s;
                p.e = sg > 0 ? p.e : -p.e;
                g = pair_value(p);
            }
            Gs[i * NP + j] = g;
        };
        // A run of interfaces per thread, upwind to downwind; the stencil (rows a ..
        // a + 6, w in upwind order from row b) slides along it, in blocks of seven
        // steps without a move while it meets neither a wrap nor an end
        const int nseg = blockDim.x >> q.logW, seg = threadIdx.x >> q.logW;
        const int j0 = seg * nout / nseg, j1 = (seg + 1) * nout / nseg;
        float w[7];
        int at = 0x40000000;  // row of w[0]
        for (int k = 0; k < j1 - j0;) {
            // interface between cells c - 1 and c; its stencil in the upwind
            // frame is centred n cells upwind (rows down to -kEdge and up to
            // L + kEdge - 1 are staged)
            const int j = sg > 0 ? j0 + k : j1 - 1 - k, c = j * every;
            int a = sg > 0 ? c - ns - 4 : c + ns - 3;
            bool inside = true;
            if (q.periodic) {
                while (a < -kEdge) a += L;
                while (a > L + 1) a -= L;
            } else {
                inside = a >= -7 && a <= L;
                a = a < -7 ? -7 : (a > L ? L : a);
            }
            const int b = sg > 0 ? a : a + 6;
            if (b == at + sg) {
#pragma unroll
                for (int m = 0; m < 6; ++m) w[m] = w[m + 1];
                w[6] = ui[(b + 6 * sg) * WP];
            } else if (b != at) {
#pragma unroll
                for (int m = 0; m < 7; ++m) w[m] = ui[(b + m * sg) * WP];
            }
            at = b;
            // (the last row read is a + 13 <= L + kEdge - 1 or a - 7 >= -kEdge)
            if (every == 1 && inside && k + 7 <= j1 - j0 && (sg > 0 ? a + 6 <= L : a - 6 >= -7)) {
                const float *v = ui + (b + 7 * sg) * WP;
#pragma unroll
                for (int m = 0; m < 7; ++m) {
                    emit(j + m * sg, vp_core::flux<float, 7, true>(sh, w[m], w[(m + 1) % 7], w[(m + 2) % 7],
                                                                   w[(m + 3) % 7], w[(m + 4) % 7], w[(m + 5) % 7],
                                                                   w[(m + 6) % 7], alpha, 1, 1));
                    w[m] = *v;
                    v += sg * WP;
                }
                at = b + 7 * sg;
                k += 7;
            } else {
                emit(j, vp_core::flux<float, 7, true>(sh, w[0], w[1], w[2], w[3], w[4], w[5], w[6], alpha, 1, 1));
                ++k;
            }
        }
        // the thread's interfaces again, the sums in double
        if (!PREFIX && over)
            for (int j = j0; j < j1; ++j) {
                const int c = j * every, d = n >= 0 ? 1 : -1;
                int a = sg > 0 ? c - ns - 4 : c + ns - 3;
                if (q.periodic) {
                    while (a < -kEdge) a += L;
                    while (a > L + 1) a -= L;
                } else {
                    a = a < -7 ? -7 : (a > L ? L : a);
                }
                const float *v = ui + (sg > 0 ? a : a + 6) * WP;
                const int s = sg * WP;
                double g = (double)vp_core::flux<float, 7, true>(sh, v[0], v[s], v[2 * s], v[3 * s], v[4 * s], v[5 * s],
                                                                 v[6 * s], alpha, 1, 1);
                v = ui + (sg > 0 ? (n >= 0 ? c - n : c) : (n >= 0 ? c : c + n)) * WP;
                for (int m = 0; m < d * n; ++m) g += (double)(d * v[m * WP]);
                Gs[i * NP + j] = sg > 0 ? g : -g;
            }
    }
    __syncthreads();
    double *out = G + l0 * nout;
    if (NP == nout && nl == W && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {  // W is even
        for (int e = 2 * (int)threadIdx.x; e < W * nout; e += 2 * (int)blockDim.x)
            *reinterpret_cast<double2 *>(out + e) = *reinterpret_cast<const double2 *>(Gs + e);
        return;
    }
    for (int k = threadIdx.x >> 5; k < nl; k += blockDim.x >> 5)
        for (int j = threadIdx.x & 31; j < nout; j += 32) out[(long long)k * nout + j] = Gs[k * NP + j];
}

// coarse state: mean over the (factor1 x factor2) fine velocity cells of a
// velocity grid [nf1][nf2] (nf2 = factor2 = 1 for one velocity dimension).
// The sum as a float pair (a conversion and an addition in double per fine
// cell took 328 us for 6.7e7 cells); quad: factor2 = 4 on 16-byte rows.
// the same sum in double, where it leaves the float range (or a cell is not finite)
__device__ __noinline__ double restrict_rare(const float *p, int nf2, int factor1, int factor2) {
    double sum = 0.0;
    for (int k = 0; k < factor1; ++k)
        for (int b = 0; b < factor2; ++b) sum += (double)p[(long long)k * nf2 + b];
    return sum;
}
__global__ void __launch_bounds__(256) k_restrict_v2(const float *__restrict__ ff, float *__restrict__ fc,
                                                     long long total, long long ncell, FastDiv nc12, FastDiv nc2,
                                                     int nf2, long long nf12,
                                                     int factor1, int factor2, int quad, double inv) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    long long x, J1;
    if (total < (1LL << 32)) {
        x = fdiv((unsigned)t, nc12);
        J1 = fdiv((unsigned)t - (unsigned)x * nc12.d, nc2);
    } else {
        x = t / ncell;
        J1 = (t - x * ncell) / nc2.d;
    }
    const long long J2 = t - x * ncell - J1 * nc2.d;
    const float *p = ff + x * nf12 + J1 * factor1 * nf2 + J2 * factor2;
    PairSum a;
    if (quad) {
#pragma unroll 4
        for (int k = 0; k < factor1; ++k) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(p + (long long)k * nf2));
            a.add(v.x);
            a.add(v.y);
            a.add(v.z);
            a.add(v.w);
        }
    } else {
        for (int k = 0; k < factor1; ++k)
            for (int b = 0; b < factor2; ++b) a.add(p[(long long)k * nf2 + b]);
    }
    double sum = pair_value(a);
    if (!isfinite(a.s)) sum = restrict_rare(p, nf2, factor1, factor2);
    fc[t] = (float)(inv != 0.0 ? sum * inv : sum / (factor1 * factor2));
}

// Samples on coarse lines: for every coarse interface with |zeta| >= zmin,
// features of the coarse stencil and the normalised target
// y = (Phi_target - Phi_CSL7) / s.  Gc: coarse-unit masses through the
// coarse interfaces ([coarse line][L + 1]).  Invalid samples get y = NaN.
// A CTA stages W lines and the lines of their velocity neighbours (STAGED; a
// line too long for shared memory is read in place) and takes their samples in
// output order, 256 at a time, lanes along a line; the 25 features leave
// through shared memory as contiguous 16-byte stores.  With a shift
// decomposition, 64-bit remainders for every stencil cell and rows of 100 bytes
// written by single threads it took 1205 us for 4.3e6 samples (430 MB).
constexpr int kSampleThreads = 256;

// a / s to 2^-47, for a result that is rounded to float: one Newton-Raphson
// correction of a times the float reciprocal, 3 FP64 instructions in place of a
// division's, which were half of the kernel's FP64 time; s outside the range in
// which neither the reciprocal nor its products leave the normal numbers takes
// the division, out of line.  Training samples of a 64 x 128 per axis 2D2V grid:
// 838 -> 811 us.
__device__ __noinline__ double ratio_rare(double a, float s) { return a / (double)s; }
__device__ __forceinline__ double ratio(double a, float s) {
    const int ex = (int)(__float_as_uint(s) >> 23 & 0xffu), ea = __double2hiint(a) >> 20 & 0x7ff;
    if ((unsigned)(ex - 27) > 200u || (unsigned)(ea - 300) > 1400u) return ratio_rare(a, s);
    const double r = widen(__frcp_rn(s)), q = __dmul_rn(a, r);
    return fma(fma(-q, widen(s), a), r, q);
}

template <bool STAGED>
__global__ void __launch_bounds__(kSampleThreads)
    k_make_samples(const float *__restrict__ fc, LineTile q, const LineShift<float> *__restrict__ tab, int kick,
                   const double *__restrict__ accel, double lo, double dvel, double dt, double h,
                   const double *__restrict__ Gc, double zmin, float *__restrict__ X, float *__restrict__ y,
                   float *__restrict__ sc, float alpha) {
    extern __shared__ __align__(16) unsigned char ssm[];
    float *xs = reinterpret_cast<float *>(ssm);  // [256][NF]
    const int L = q.L, W = q.W, P = (L + 2 * kEdge) | 1;
    float *tile = xs + kSampleThreads * NF;      // STAGED: [3][W][P]: the lines, +, - neighbours
    const long long l0 = (long long)blockIdx.x * W;
    const int nl = (int)(q.lines - l0 < W ? q.lines - l0 : W);
    __shared__ LinePos pos;
    // velocity neighbours: 1: class + 1 is the + one (larger |v|), 2: class + 1
    // is in the box, 4: class - 1 is
    __shared__ int nbr[kTileLines];
    place_lines(q, l0, nl, pos);
    __syncthreads();
    for (int i = threadIdx.x; i < nl; i += blockDim.x) {
        const unsigned cls = pos.cls[i];
        nbr[i] = kick ? 0
                      : (vp_core::cell_centre(lo, dvel, (int)cls) >= 0.0 ? 1 : 0) | (cls + 1 < q.cmod ? 2 : 0) |
                            (cls > 0 ? 4 : 0);
    }
    __syncthreads();
    if (STAGED) {
        for (int k = 0; k < 3; ++k) {  // the lines, then class + 1 and class - 1
            float *d = tile + (size_t)k * W * P + kEdge;
            stage_lines(fc, q, pos, nl, k == 0 ? 0 : (k == 1 ? 1 : -1) * q.cdiv,
                        [&](int i) { return k == 0 || (nbr[i] & (k == 1 ? 2 : 4)); },
                        [&](int i, int row) { return d + i * P + row; });
        }
        vp_tma::cp_async_wait_all();
        __syncthreads();
    }
    const int ns = nl * (L + 1);
    const long long t0 = l0 * (L + 1);
    for (int b0 = 0; b0 < ns; b0 += kSampleThreads) {
        const int t = b0 + threadIdx.x;
        float x[NF];
        if (t < ns) {
            const int i = t / (L + 1), j = t - i * (L + 1);  // line, interface between cells j - 1 and j
            const long long line = l0 + i;
            const unsigned cls = pos.cls[i];
            const LineShift<float> sh = tab[cls];
            bool none = q.periodic && j == L;
            if (zmin > 0.0 && !none) {
                const double speed = kick ? accel[cls] : vp_core::cell_centre(lo, dvel, (int)cls);
                const double s_full = speed * dt / h;
                none = fabs(s_full - round(s_full)) < zmin;
            }
            if (none) {
#pragma unroll
                for (int k = 0; k < NF; ++k) x[k] = 0.f;
                y[t0 + t] = __int_as_float(0x7fc00000);
                if (sc) sc[t0 + t] = 0.f;
            } else {
                const int sg = sh.sigma, n = sh.n * sg;
                // row r of the line, or of the neighbour of class + 1 / - 1
                const float *own = tile + kEdge + i * P, *base = fc + pos.base[i];
                auto cell = [&](int nb, int r) -> float {
                    if (STAGED) return own[(nb == 0 ? 0 : (nb > 0 ? 1 : 2)) * (W * P) + r];
                    if (nb && !(nbr[i] & (nb > 0 ? 2 : 4))) return 0.f;
                    if (q.periodic) r = wrap_row(r, L);
                    else if (r < 0 || r >= L) return 0.f;
                    return base[(long long)r * q.inner + nb * q.cdiv];
                };
                // stencil cells: rows a .. a + 7, in upwind order by sg
                const int nsh = q.periodic ? n % L : (n < -2 * L - 8 ? -2 * L - 8 : (n > 2 * L + 8 ? 2 * L + 8 : n));
                int a = sg > 0 ? j - nsh - 4 : j + nsh - 4;
                a = q.periodic ? wrap_row(a, L) : (a < -8 ? -8 : (a > L ? L : a));
                float u[8], unp[8], unm[8];
                const int sp = (nbr[i] & 1) ? 1 : -1;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int r = a + (sg > 0 ? k : 7 - k);
                    u[k] = cell(0, r);
                    unp[k] = cell(sp, r);
                    unm[k] = cell(-sp, r);
                }
                // whole cells swept in the upwind frame, signed (n < 0 when the
                // integer shift opposes the fractional one)
                double whole = 0.0;
                int k = sg > 0 ? (n >= 0 ? j - n : j) : (n >= 0 ? j : j + n);
                int r = q.periodic ? k % L : k;
                r = q.periodic && r < 0 ? r + L : r;
                for (int m = n >= 0 ? n : -n; m > 0; --m) {
                    if (q.periodic || (r >= 0 && r < L)) whole += widen(cell(0, r));
                    ++r;
                    if (q.periodic && r == L) r = 0;
                }
                if (n < 0) whole = -whole;
                const double gc = Gc[line * (L + 1) + j];
                const double g = sg > 0 ? gc : -gc;
                // coarse fractional mass as the plain sweep computes it: CSL7, then MP
                float phi = sh.w[0] * u[0];
#pragma unroll
                for (int m = 1; m < 7; ++m) phi = fmaf(sh.w[m], u[m], phi);
                phi = vp_core::mp_limit(phi, u[1], u[2], u[3], u[4], u[5], alpha);
                const float s = net_features(u, unp, unm, sh.nu, x);
                y[t0 + t] = (float)ratio(g - whole - widen(sh.nu) * widen(phi), s);
                if (sc) sc[t0 + t] = s;
            }
#pragma unroll
            for (int k = 0; k < NF; ++k) xs[threadIdx.x * NF + k] = x[k];
        }
        __syncthreads();
        const int m = (ns - b0 < kSampleThreads ? ns - b0 : kSampleThreads) * NF;
        float *out = X + (t0 + b0) * NF;
        if ((reinterpret_cast<uintptr_t>(out) & 15) == 0) {
            for (int e = 4 * threadIdx.x; e + 3 < m; e += 4 * kSampleThreads)
                *reinterpret_cast<float4 *>(out + e) = *reinterpret_cast<const float4 *>(xs + e);
            for (int e = (m & ~3) + threadIdx.x; e < m; e += kSampleThreads) out[e] = xs[e];
        } else {
            for (int e = threadIdx.x; e < m; e += kSampleThreads) out[e] = xs[e];
        }
        __syncthreads();
    }
}

// cell pairs of the training loss: the residual of the cell between
// interfaces l and r is (s_r (g_r - y_r) - s_l (g_l - y_l)) / max(s_l, s_r),
// so the pair's coefficients are (-s_l / m, s_r / m), m = max(s_l, s_r); the
// draw weight of the pair is m^importance (1 for importance 0)
__global__ void k_pair_coefs(const float *__restrict__ sc, const long long *__restrict__ li,
                             const long long *__restrict__ ri, long long n, double importance,
                             float *__restrict__ coef, double *__restrict__ weight) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double sl = sc[li[t]], sr = sc[ri[t]];
    const double m = sl > sr ? sl : sr;
    coef[2 * t] = (float)(-(sl / m));
    coef[2 * t + 1] = (float)(sr / m);
    if (weight) weight[t] = importance > 0.0 ? pow(m, importance) : 1.0;
}

// coarse-interface masses from fine ones: mean over `group` fine lines of
// every fine value, scaled by `scale` (fine -> coarse cell units)
// (32-bit indices; a division only where 1 / group is not exact)
__global__ void __launch_bounds__(256) k_group_mean(const double *__restrict__ Gf, long long total, int nout,
                                                    FastDiv fd_nout, const long long *__restrict__ map, int group,
                                                    double scale, double inv, double *__restrict__ Gc) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const long long cl = total < (1LL << 32) ? (long long)fdiv((unsigned)t, fd_nout) : t / nout;
    const int j = (int)(t - cl * nout);
    const long long *m = map + cl * group;
    double s = 0.0;
#pragma unroll 8
    for (int g = 0; g < group; ++g) s += Gf[m[g] * nout + j];
    Gc[t] = inv != 0.0 ? scale * s * inv : scale * s / group;
}

// ---- inference: the learned coarse sweep, network on the tensor cores -------------------
//
// A CTA stages a tile of lines of the drift along x_d in shared memory: all L
// cells of each line, for every velocity index j of the axis v_d (the line
// class) times a block of the other indices, so that the velocity neighbours
// of every line (j +- 1, the +/- lines of the features) are in the tile and no
// other CTA reads the tile's lines: the update is written to f in place,
// without a snapshot.  Each lane then walks one line upwind -> downwind as the
// plain line walker does (8-cell windows of the line and of its velocity
// difference and curvature in registers, one new row per interface, the MP
// curvature and d^{M4} carried), and at every interface the warp's 32 lanes
// form one 32-row feature tile for the network on the tensor cores.  The
// interface mass (plain MP mass plus s g, MP bounds when asked, PP) leaves the
// upwind cell and enters the next, so each cell is written once:
// f' = (u - M_out) + M_in.

constexpr int kTcThreads = 128;  // one line per thread, one 128-row MMA operand per interface step

// tile of a learned sweep: columns col = (g cmod + j) T + t hold the line with
// inner index c = c_tile + g cmod cdiv + j cdiv + t (class j); tiles per outer
// index: (inner / (G cmod cdiv)) (cdiv / T)
struct LTile {
    long long outer, inner, cdiv, cmod;
    int L, T, G, NC, pitch;  // NC = G cmod T columns, row pitch in floats
    long long tpo;           // tiles per outer index
    long long tblocks;       // t blocks per group block: cdiv / T
};

// Network operands for the tensor cores, prepared once per call from the
// FP32 master weights: W1, W2, W3 (32 outputs x 48 inputs) and w4 (row 0 of a
// 16 x 48 matrix) as bf16 in the canonical K-major layout.  Inputs 0-31 are
// the layer's inputs (W1 zero beyond its 25 features); every A row carries
// the constant 1 in columns 32 and 33, and the operands hold the bias there
// as a bf16 pair, b = bf16(b) + bf16(b - bf16(b)), so the accumulator starts
// from the bias to 16 significant bits and no epilogue adds it.
constexpr int kOpW = 32 * vp_umma::kK * 2;    // bytes of one 32-row bf16 operand
constexpr int kOpW4 = 16 * vp_umma::kK * 2;   // 16 rows
constexpr int kOpBytes = 3 * kOpW + kOpW4;
constexpr int kOpAlloc = (kOpBytes + 127) / 128 * 128;

__global__ void k_net_umma(const float *__restrict__ wts, unsigned char *__restrict__ out) {
    constexpr int K = vp_umma::kK;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 3 * 32 * K + 16 * K; e += gridDim.x * blockDim.x) {
        int layer, n, k;
        if (e < 3 * 32 * K) {
            layer = e / (32 * K);
            n = (e / K) % 32;
            k = e % K;
        } else {
            layer = 3;
            n = (e - 3 * 32 * K) / K;
            k = (e - 3 * 32 * K) % K;
        }
        const int kin = layer == 0 ? NF : H;
        float w = 0.f, b = 0.f;
        if (layer < 3) {
            const int base = layer == 0 ? OFF_W1 : (layer == 1 ? OFF_W2 : OFF_W3);
            w = k < kin ? wts[base + n * kin + k] : 0.f;
            b = wts[(layer == 0 ? OFF_B1 : (layer == 1 ? OFF_B2 : OFF_B3)) + n];
        } else if (n == 0) {
            w = k < H ? wts[OFF_W4 + k] : 0.f;
            b = wts[OFF_B4];
        }
        const float bh = __bfloat162float(__float2bfloat16_rn(b));
        const float v = k < 32 ? w : k == 32 ? bh : k == 33 ? b - bh : 0.f;
        const uint32_t off = (uint32_t)(layer * kOpW) + vp_umma::kmajor_offset(n, k);
        *reinterpret_cast<__nv_bfloat16 *>(out + off) = __float2bfloat16_rn(v);
    }
}

constexpr int kABytes = 128 * vp_umma::kK * 2;  // one 128 x 48 bf16 feature operand
// interfaces per line in one network batch: three operands and the weights
// take 46.5 KB of shared memory and 128 tensor-memory columns, so four CTAs
// share an SM (all 512 columns)
constexpr int kLC = 3;
// tensor-memory columns of a CTA: the power of two >= 32 that holds LC
// accumulators of 32 columns
__host__ __device__ constexpr uint32_t tmem_cols(int lc) {
    return lc <= 1 ? 32u : (lc <= 2 ? 64u : (lc <= 4 ? 128u : 256u));
}

// bf16 columns 0-31 of row r (in w) of an operand in the canonical layout
__device__ __forceinline__ void store_row(unsigned char *op, int r, const uint32_t (&w)[16]) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
        *reinterpret_cast<uint4 *>(op + vp_umma::kmajor_offset(r, 8 * kk)) =
            make_uint4(w[4 * kk], w[4 * kk + 1], w[4 * kk + 2], w[4 * kk + 3]);
}

// The three hidden layers and the output layer for `nb` operands of 128
// feature rows (operand b at A + b kABytes, accumulator columns 32 b .. 32 b
// + 31), on the tensor cores: one thread issues each layer's MMAs (three
// k-blocks of 16) and commits them to the mbarrier; every thread then reads
// its own row back from tensor memory, applies ReLU, rounds to bf16 and
// writes it as the next layer's A row.  Returns g of this thread's row of
// each operand.  Bounded waits: on a timeout the status word is set.
template <int LC>
__device__ __forceinline__ void net_tc(unsigned char *A, const unsigned char *ops, uint32_t tmem, uint64_t *bar,
                                       uint32_t &phase, int nb, float (&g)[LC], int *status) {
    const int warp = threadIdx.x >> 5;
    const uint32_t a_s = vp_tma::saddr(A), w_s = vp_tma::saddr(ops);
    const uint32_t tl = tmem + ((uint32_t)(32 * warp) << 16);
    for (int layer = 0; layer < 4; ++layer) {
        vp_umma::fence_proxy_async();
        vp_umma::fence_before_sync();
        __syncthreads();
        if (threadIdx.x == 0) {
            vp_umma::fence_after_sync();
            const uint32_t idesc = vp_umma::idesc_bf16_f32(128, layer < 3 ? 32 : 16);
            const uint64_t bd = vp_umma::smem_desc(w_s + (uint32_t)(layer * kOpW), 128, vp_umma::kSBO);
            for (int b = 0; b < nb; ++b) {
                const uint64_t ad = vp_umma::smem_desc(a_s + (uint32_t)(b * kABytes), 128, vp_umma::kSBO);
#pragma unroll
                for (int s = 0; s < vp_umma::kK / 16; ++s)  // 256 bytes per k-block: 16 to the address field
                    vp_umma::mma_bf16(tmem + (uint32_t)(32 * b), ad + (uint64_t)(16 * s), bd + (uint64_t)(16 * s),
                                      idesc, (uint32_t)s);
            }
            vp_umma::commit(bar);
        }
        const bool done = vp_tma::mbar_wait(bar, phase, 1u << 24);
        phase ^= 1u;
        if (!done) atomicExch(status, VP_ETIMEOUT);
        vp_umma::fence_after_sync();
        if (layer < 3) {
            for (int b = 0; b < nb; ++b) {
                float v[32];
                vp_umma::ld32(tl + (uint32_t)(32 * b), v);
                uint32_t w[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = pack_relu_bf16(v[2 * i], v[2 * i + 1]);
                store_row(A + b * kABytes, threadIdx.x, w);
            }
        } else {
#pragma unroll
            for (int b = 0; b < LC; ++b) g[b] = b < nb ? vp_umma::ld1(tl + (uint32_t)(32 * b)) : 0.f;
        }
    }
}

// Reads f^n (fin, not written during the launch) through L2 and writes the
// updated lines to fout; a thread reads its line and the two lines of the
// neighbouring velocity cells row by row as it walks.
template <bool PERIODIC, int LC>
__global__ void __launch_bounds__(kTcThreads) k_learned_walk(const float *__restrict__ fin, float *__restrict__ fout,
                                                             LTile tl, const LineShift<float> *__restrict__ tab,
                                                             const uint4 *__restrict__ netops, double lo,
                                                             double dvel, float alpha, int mode,
                                                             int *__restrict__ status) {
    extern __shared__ __align__(1024) unsigned char tsm[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    unsigned char *A = tsm;                                // LC operands of 128 x 48 bf16
    unsigned char *ops = tsm + LC * kABytes;               // W1 W2 W3 w4, biases
    const int L = tl.L, NC = tl.NC, T = tl.T;
    const int cmod = (int)tl.cmod;
    const long long o = (long long)blockIdx.x / tl.tpo;
    const long long tin = (long long)blockIdx.x - o * tl.tpo;
    const long long gb = tin / tl.tblocks, tb = tin - gb * tl.tblocks;
    // inner index of column col
    auto col_c = [&](int col) -> long long {
        const int t = col % T, jg = col / T;
        const int j = jg % cmod, g = jg / cmod;
        return (gb * tl.G + g) * tl.cmod * tl.cdiv + (long long)j * tl.cdiv + tb * T + t;
    };
    const long long obase = o * (long long)L * tl.inner;
    // phase 0: network operands, tensor memory, mbarrier
    for (int e = threadIdx.x; e < kOpAlloc / 16; e += blockDim.x)
        reinterpret_cast<uint4 *>(ops)[e] = netops[e];
    // columns 32-47 of every A row: 1, 1 (the bias pair), then zeros
    for (int b = 0; b < LC; ++b)
#pragma unroll
        for (int kk = 4; kk < vp_umma::kK / 8; ++kk)
            *reinterpret_cast<uint4 *>(A + b * kABytes + vp_umma::kmajor_offset(threadIdx.x, 8 * kk)) =
                kk == 4 ? make_uint4(pack2(1.f, 1.f), 0u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    if (threadIdx.x < 32) vp_umma::tmem_alloc(&tslot, tmem_cols(LC));
    if (threadIdx.x == 0) {
        vp_tma::mbar_init(&bar, 1);
        vp_tma::fence_mbar_init();
    }
    vp_umma::fence_before_sync();
    __syncthreads();
    vp_umma::fence_after_sync();
    const uint32_t tmem = tslot;
    uint32_t phase = 0;
    const int col = threadIdx.x;
    const bool ok = col < NC;
    const int colc = ok ? col : 0;
    // the line's shift and its velocity neighbours (+: larger |v|)
    const int j = (colc / T) % cmod;
    const LineShift<float> sh = tab[j];
    const int sg = sh.sigma;
    const float nu = sh.nu;
    const int sp = vp_core::cell_centre(lo, dvel, j) >= 0.0 ? 1 : -1;
    const int cp = (j + sp >= 0 && j + sp < cmod) ? colc + sp * T : -1;
    const int cm = (j - sp >= 0 && j - sp < cmod) ? colc - sp * T : -1;
    int n = sh.n;
    if (PERIODIC) {  // the shift modulo L
        n %= L;
        if (n < 0) n += L;
    }
    // source row of the upwind cell of interface 0 (the cell before the
    // walk's first cell), unwrapped for zero-inflow lines
    const int q = (sg > 0 ? 0 : L - 1) - n - sg;
    auto wrap = [&](int r) -> int {
        if (PERIODIC) {
            r %= L;
            if (r < 0) r += L;
        }
        return r;
    };
    // the line and its velocity neighbours in f^n (row r at r inner)
    const float *pu = fin + obase + col_c(colc);
    const float *pp = fin + obase + col_c(cp >= 0 ? cp : colc);
    const float *pm = fin + obase + col_c(cm >= 0 ? cm : colc);
    // cell value, velocity difference and velocity curvature at row r (wrapped
    // for periodic lines; outside [0, L) zero for zero-inflow lines)
    auto fetch_w = [&](int r, float &u, float &dv, float &cv) {
        const bool in = ok && (PERIODIC || (r >= 0 && r < L));
        const long long o = (long long)r * tl.inner;
        u = in ? __ldg(pu + o) : 0.f;
        const float up = in && cp >= 0 ? __ldg(pp + o) : 0.f;
        const float um = in && cm >= 0 ? __ldg(pm + o) : 0.f;
        dv = up - um;
        cv = fmaf(0.5f, up + um, -u);
    };
    float u[8], dv[8], cv[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) fetch_w(wrap(q + (m - 3) * sg), u[m], dv[m], cv[m]);
    // the row entering the window after interface k: q + (5 + k) sg, wrapped
    // incrementally.  Rows enter as raw values (u, u+, u-) loaded one batch
    // ahead: the next batch's rows are requested before this batch's network
    // round trips, which hide the L2 latency.
    int rn = wrap(q + 5 * sg);
    auto load_raw = [&](float &a, float &ap, float &am) {
        const bool in = ok && (PERIODIC || (rn >= 0 && rn < L));
        const long long o = (long long)rn * tl.inner;
        a = in ? __ldg(pu + o) : 0.f;
        ap = in && cp >= 0 ? __ldg(pp + o) : 0.f;
        am = in && cm >= 0 ? __ldg(pm + o) : 0.f;
        rn += sg;
        if (PERIODIC) {
            rn = rn == L ? 0 : rn;
            rn = rn < 0 ? L - 1 : rn;
        }
    };
    float ru[LC], rp[LC], rm[LC];
#pragma unroll
    for (int b = 0; b < LC; ++b) load_raw(ru[b], rp[b], rm[b]);
    // MP carries: curvature of the upwind cell, d^{M4} at its upwind face
    float dc = vp_core::curv(u[2], u[3], u[4]);
    float m4m = vp_core::dm4(vp_core::curv(u[1], u[2], u[3]), dc);
    float Min = 0.f;
    const long long cbase = obase + col_c(colc);
#pragma unroll 1
    for (int k0 = 0; k0 <= L; k0 += LC) {
        const int nb = L + 1 - k0 < LC ? L + 1 - k0 : LC;
        float xu[LC], xp[LC], xm[LC];  // the next batch's rows
#pragma unroll
        for (int b = 0; b < LC; ++b) load_raw(xu[b], xp[b], xm[b]);
        float Mp[LC], sc[LC], mlo[LC], mhi[LC], u3[LC], u4[LC];
#pragma unroll
        for (int b = 0; b < LC; ++b) {
            if (b >= nb) break;
            // plain mass of interface k0 + b (CSL7, MP bounds as a clamp)
            const float dp = vp_core::curv(u[3], u[4], u[5]);
            const float m4p = vp_core::dm4(dc, dp);
            float phi = sh.w[0] * u[0];
#pragma unroll
            for (int m = 1; m < 7; ++m) phi = fmaf(sh.w[m], u[m], phi);
            vp_core::mp_lohi_carried(u[2], u[3], u[4], alpha, m4m, m4p, mlo[b], mhi[b]);
            Mp[b] = vp_core::mul_rn(nu, fminf(fmaxf(phi, mlo[b]), mhi[b]));
            u3[b] = u[3];
            u4[b] = u[4];
            // feature row (columns 0-7 stencil, 8-15 velocity difference,
            // 16-23 velocity curvature, 24 nu, 25-31 zero), as net_features
            float s = 0.f;
#pragma unroll
            for (int m = 0; m < 8; ++m) s = fmaxf(s, fabsf(u[m]));
            s += 1e-30f;
            sc[b] = s;
            const float inv = 1.0f / s;
            const float hinv = 0.5f * inv;
            uint32_t w[16];
#pragma unroll
            for (int m = 0; m < 4; ++m) w[m] = pack2((u[2 * m] - u[3]) * inv, (u[2 * m + 1] - u[3]) * inv);
            w[1] = pack2((u[2] - u[3]) * inv, 0.f);
#pragma unroll
            for (int m = 0; m < 4; ++m) w[4 + m] = pack2(dv[2 * m] * hinv, dv[2 * m + 1] * hinv);
#pragma unroll
            for (int m = 0; m < 4; ++m) w[8 + m] = pack2(cv[2 * m] * inv, cv[2 * m + 1] * inv);
            w[12] = pack2(nu, 0.f);
            w[13] = w[14] = w[15] = 0u;
            store_row(A + b * kABytes, threadIdx.x, w);
            // advance the window and the MP carries
            dc = dp;
            m4m = m4p;
            const float un = ru[b], dvn = rp[b] - rm[b], cvn = fmaf(0.5f, rp[b] + rm[b], -un);
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                u[m] = u[m + 1];
                dv[m] = dv[m + 1];
                cv[m] = cv[m + 1];
            }
            u[7] = un;
            dv[7] = dvn;
            cv[7] = cvn;
        }
        float g[LC];
        net_tc<LC>(A, ops, tmem, &bar, phase, nb, g, status);
#pragma unroll
        for (int b = 0; b < LC; ++b) {
            ru[b] = xu[b];
            rp[b] = xp[b];
            rm[b] = xm[b];
        }
#pragma unroll
        for (int b = 0; b < LC; ++b) {
            if (b >= nb) break;
            float M = fmaf(sc[b], g[b], Mp[b]);
            if (mode == 2) M = fminf(fmaxf(M, vp_core::mul_rn(nu, mlo[b])), vp_core::mul_rn(nu, mhi[b]));
            M = vp_core::pp_clamp(M, vp_core::half_rd(u3[b]), vp_core::half_rd(u4[b]));
            // the cell whose source is u3 takes M in from the previous interface
            const int k = k0 + b;
            if (ok && k >= 1) {
                const int i = sg > 0 ? k - 1 : L - k;
                fout[cbase + (long long)i * tl.inner] = (u3[b] - M) + Min;
            }
            Min = M;
        }
    }
    vp_umma::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) {
        vp_umma::fence_after_sync();
        vp_umma::tmem_dealloc(tmem, tmem_cols(LC));
    }
}

}  // namespace

// ---- host entry points ------------------------------------------------------------------

extern "C" {

int vp_net_grad(const float *X, const float *y, const float *coef, long long nsamp, int group, const float *wts,
                float *grad, float *loss, void *stream) {
    if (!X || !y || !wts || !grad || !loss || nsamp < 1 || (group != 1 && group != 2) || nsamp % group)
        return VP_EINVAL;
    // SMs of the device, looked up (and the kernel's shared memory set) by the
    // first call on it: a training step is three short launches
    static std::atomic<int> sm_count[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return VP_ECUDA;
    int sms = sm_count[dev].load(std::memory_order_acquire);
    if (!sms) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaFuncSetAttribute(k_net_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrainSmem) !=
                cudaSuccess)
            return VP_ECUDA;
        sm_count[dev].store(sms, std::memory_order_release);
    }
    const long long tiles = (nsamp + 15) / 16;
    const long long blocks = tiles < sms ? tiles : sms;  // one CTA per SM at most
    k_net_grad<<<(unsigned)blocks, kTrainThreads, kTrainSmem, static_cast<cudaStream_t>(stream)>>>(
        X, y, coef, wts, nsamp, group, grad, loss);
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

int vp_net_adam(float *wts, float *m, float *v, float *grad, int step, float lr, void *stream) {
    if (!wts || !m || !v || !grad || step < 1 || !(lr > 0.f)) return VP_EINVAL;
    const float b1 = 0.9f, b2 = 0.999f;
    const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
    k_adam<<<(NPARAM + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(wts, m, v, grad, NPARAM, lr, b1,
                                                                               b2, 1e-8f, bc1, bc2);
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

}  // extern "C"

// geometry helpers shared with the context-level entry points below
namespace {
struct LineGeo {
    long long outer, inner;
    int L, periodic, kick, from_inner;
    long long cdiv, cmod;
    double lo, dvel, h;
};

LineGeo line_geo(const vp_grid &g, long long NX, long long NV, int kick, int dim) {
    LineGeo q{};
    if (!kick) {
        long long outer = 1, inner = NV, vstride = 1;
        for (int k = 0; k < dim; ++k) outer *= g.nx[k];
        for (int k = dim + 1; k < g.dx; ++k) inner *= g.nx[k];
        for (int k = dim + 1; k < g.dv; ++k) vstride *= g.nv[k];
        q.outer = outer;
        q.inner = inner;
        q.L = g.nx[dim];
        q.periodic = g.xbc == VP_BC_PERIODIC;
        q.from_inner = 1;
        q.cdiv = vstride;
        q.cmod = g.nv[dim];
        q.h = (g.xhi[dim] - g.xlo[dim]) / g.nx[dim];
    } else {
        long long vouter = 1, inner = 1;
        for (int k = 0; k < dim; ++k) vouter *= g.nv[k];
        for (int k = dim + 1; k < g.dv; ++k) inner *= g.nv[k];
        q.outer = NX * vouter;
        q.inner = inner;
        q.L = g.nv[dim];
        q.periodic = 0;
        q.from_inner = 0;
        q.cdiv = vouter;
        q.cmod = 1;
        q.h = (g.vhi[dim] - g.vlo[dim]) / g.nv[dim];
    }
    q.kick = kick;
    q.lo = g.vlo[dim];
    q.dvel = (g.vhi[dim] - g.vlo[dim]) / g.nv[dim];
    return q;
}

LineTile line_tile(const LineGeo &q) {
    LineTile t{};
    t.lines = q.outer * q.inner;
    t.inner = q.inner;
    t.L = q.L;
    t.periodic = q.periodic;
    t.from_inner = q.from_inner;
    t.cdiv = q.cdiv;
    t.cmod = (unsigned)q.cmod;
    t.prepare();
    return t;
}
void set_width(LineTile &t, int W) {
    t.W = W;
    t.logW = 0;
    while ((1 << t.logW) < W) ++t.logW;
}
}  // namespace

int vp_learned_prepare(vp_ctx *c) {
    if (c->learned_ready) return VP_OK;
    if (!c->d_netfrag) VP_CUDA_TRY(c, cudaMalloc(&c->d_netfrag, kOpAlloc));
    // the updated lines of a learned sweep (copied back into f after the walk)
    if (!c->d_learn_out) VP_CUDA_TRY(c, cudaMalloc(&c->d_learn_out, (size_t)c->ncell * sizeof(float)));
    VP_CUDA_TRY(c, cudaFuncSetAttribute(k_learned_walk<true, kLC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        200 * 1024));
    VP_CUDA_TRY(c, cudaFuncSetAttribute(k_learned_walk<false, kLC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        200 * 1024));
    c->learned_ready = 1;
    return VP_OK;
}

// one learned drift along dim from fin (f^n, not written) to fout; with
// net = true the network operands are made from wts first (a stage of
// several drifts with one network makes them once)
int vp_learned_drift_io(vp_ctx *c, int dim, double dt, const float *wts, int use_net, const float *fin,
                        float *fout, bool net, bool tab_ready) {
    const LineGeo q = line_geo(c->g, c->NX, c->NV, 0, dim);
    // tile: every class j of its lines times a block of the other indices,
    // about 128 lines (columns)
    LTile tl{};
    tl.outer = q.outer;
    tl.inner = q.inner;
    tl.cdiv = q.cdiv;
    tl.cmod = q.cmod;
    tl.L = q.L;
    const long long NG = q.inner / (q.cmod * q.cdiv);
    const int target = 128;
    if (q.cmod > kTcThreads)
        return vp_fail(c, VP_ENOTSUP, "more than %d velocity cells on the sweep's axis", kTcThreads);
    if (q.cmod * q.cdiv <= target) {
        tl.T = (int)q.cdiv;
        long long G = target / (q.cmod * q.cdiv);
        while (G > 1 && NG % G) --G;
        tl.G = (int)(G < 1 ? 1 : G);
    } else {
        tl.G = 1;
        long long T = target / q.cmod;
        if (T < 1) T = 1;
        while (T > 1 && q.cdiv % T) --T;
        tl.T = (int)T;
    }
    tl.NC = (int)(tl.G * q.cmod * tl.T);
    tl.pitch = 0;
    tl.tblocks = q.cdiv / tl.T;
    tl.tpo = (NG / tl.G) * tl.tblocks;
    const int threads = kTcThreads;  // one 128-row operand: a thread per row, rows >= NC are idle
    const size_t smem = (size_t)kLC * kABytes + kOpAlloc;
    const long long blocks = q.outer * tl.tpo;
    if (blocks >= (1LL << 31)) return vp_fail(c, VP_ENOTSUP, "learned sweep has too many tiles");
    // the drifts' shifts: with the network's operands, once for a stage
    int rc = tab_ready ? VP_OK : vp_launch_shift_tables(c, 0, 1u << dim, dt, nullptr);
    if (rc != VP_OK) return rc;
    if (net) {
        k_net_umma<<<(4 * 32 * vp_umma::kK + 255) / 256, 256, 0, c->stream>>>(wts, static_cast<unsigned char *>(c->d_netfrag));
        c->launches++;
    }
    const LineShift<float> *tab = static_cast<const LineShift<float> *>(c->d_shift) + dim * c->shift_cap;
    const uint4 *ops = static_cast<const uint4 *>(c->d_netfrag);
    if (q.periodic)
        k_learned_walk<true, kLC><<<(unsigned)blocks, threads, smem, c->stream>>>(
            fin, fout, tl, tab, ops, q.lo, q.dvel, (float)c->g.alpha, use_net, c->d_status);
    else
        k_learned_walk<false, kLC><<<(unsigned)blocks, threads, smem, c->stream>>>(
            fin, fout, tl, tab, ops, q.lo, q.dvel, (float)c->g.alpha, use_net, c->d_status);
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

extern "C" {

int vp_learned_sweep(vp_ctx *c, int kick, int dim, double dt, const double *accel_dev, const float *wts,
                     int use_net, const float *f_snap) {
    (void)f_snap;  // the walk reads f^n as it is and writes the new lines to a buffer of its own
    if (!c || !c->f) return VP_EINVAL;
    if (c->g.precision != VP_F32 || c->g.order != 7)
        return vp_fail(c, VP_ENOTSUP, "the learned sweep runs on FP32 CSL7 grids");
    if (use_net < 0 || use_net > 2) return vp_fail(c, VP_EINVAL, "use_net must be 0, 1 or 2");
    if (use_net && kick) return vp_fail(c, VP_ENOTSUP, "the learned correction applies to spatial sweeps");
    if (dim < 0 || dim >= c->g.dx || (kick && !accel_dev) || (use_net && !wts) || !std::isfinite(dt))
        return vp_fail(c, VP_EINVAL, "bad learned-sweep arguments");
    if (!use_net) return kick ? vp_kick_sweep(c, dim, dt, accel_dev) : vp_drift_sweep(c, dim, dt);
    int rc = vp_learned_prepare(c);
    if (rc != VP_OK) return rc;
    float *fout = static_cast<float *>(c->d_learn_out);
    if ((rc = vp_learned_drift_io(c, dim, dt, wts, use_net, static_cast<const float *>(c->f), fout, true,
                                  false)))
        return rc;
    VP_CUDA_TRY(c, cudaMemcpyAsync(c->f, fout, (size_t)c->ncell * sizeof(float), cudaMemcpyDeviceToDevice,
                                   c->stream));
    return VP_OK;
}

int vp_fine_flux(vp_ctx *c, int kick, int dim, double dt, const double *accel_dev, int every,
                 double *G_dev) {
    if (!c || !c->f || !G_dev || every < 1) return VP_EINVAL;
    if (c->g.precision != VP_F32 || c->g.order != 7)
        return vp_fail(c, VP_ENOTSUP, "fine fluxes are computed for FP32 CSL7 grids");
    if (dim < 0 || dim >= c->g.dx || (kick && !accel_dev)) return vp_fail(c, VP_EINVAL, "bad fine-flux arguments");
    const LineGeo q = line_geo(c->g, c->NX, c->NV, kick, dim);
    if (q.L % every) return vp_fail(c, VP_EINVAL, "line length must be a multiple of `every`");
    if ((size_t)q.L * 64 * sizeof(double) > 200 * 1024) return vp_fail(c, VP_ENOTSUP, "line too long");
    LineTile t = line_tile(q);
    // whole-cell parts: a drift's longest is known here, a kick's only on the device
    const double vmax = std::fmax(std::fabs(c->g.vlo[dim]), std::fabs(c->g.vhi[dim]));
    const bool prefix = kick || !(vmax * std::fabs(dt) / q.h + 1.0 < kFewCells);
    const int nout = q.L / every + 1;
    auto bytes = [&](int W) {
        return (size_t)W * (nout | 1) * sizeof(double) + (prefix ? (size_t)(q.L + 1) * W * sizeof(double) : 0) +
               (size_t)(q.L + 2 * kEdge) * (W + 1) * sizeof(float);
    };
    int W = kTileLines;
    while (W > 8 && bytes(W) > 72 * 1024) W /= 2;  // three CTAs per SM
    set_width(t, W);
    const size_t smem = bytes(W);
    const int rc = vp_launch_shift_tables_f32(c, kick, 1u << dim, dt, accel_dev);
    if (rc) return rc;
    const LineShift<float> *tab = static_cast<const LineShift<float> *>(c->d_shift) + dim * c->shift_cap;
    const unsigned blocks = (unsigned)((t.lines + t.W - 1) / t.W);
    const bool quad = t.inner % 4 == 0 && (reinterpret_cast<uintptr_t>(c->f) & 15) == 0;
    auto launch = [&](auto kernel) -> int {
        VP_CUDA_TRY(c, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        kernel<<<blocks, 256, smem, c->stream>>>(static_cast<const float *>(c->f), t, tab, every, G_dev,
                                                 (float)c->g.alpha);
        return VP_OK;
    };
    const int lrc = prefix ? (quad ? launch(k_fine_flux<true, true>) : launch(k_fine_flux<true, false>))
                           : (quad ? launch(k_fine_flux<false, true>) : launch(k_fine_flux<false, false>));
    if (lrc) return lrc;
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

int vp_restrict_velocity(const float *f_fine, float *f_coarse, long long NX, int nf1, int nf2, int factor1,
                         int factor2, void *stream) {
    if (!f_fine || !f_coarse || factor1 < 1 || factor2 < 1 || nf1 < 1 || nf2 < 1 || nf1 % factor1 || nf2 % factor2)
        return VP_EINVAL;
    const int nc1 = nf1 / factor1, nc2 = nf2 / factor2;
    const long long ncell = (long long)nc1 * nc2, n = NX * ncell;
    const int quad = factor2 == 4 && (reinterpret_cast<uintptr_t>(f_fine) & 15) == 0, ff = factor1 * factor2;
    const double inv = (ff & (ff - 1)) == 0 ? 1.0 / ff : 0.0;  // exact
    k_restrict_v2<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        f_fine, f_coarse, n, ncell, make_fastdiv(n < (1LL << 32) ? (unsigned)ncell : 1u), make_fastdiv((unsigned)nc2), nf2,
        (long long)nf1 * nf2, factor1, factor2, quad, inv);
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

int vp_pair_coefs(const float *sc, const long long *li, const long long *ri, long long n, double importance,
                  float *coef, double *weight, void *stream) {
    if (!sc || !li || !ri || !coef || n < 0 || !(importance >= 0.0)) return VP_EINVAL;
    if (n == 0) return VP_OK;
    k_pair_coefs<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(sc, li, ri, n,
                                                                                            importance, coef, weight);
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

int vp_group_mean(const double *G_fine, long long n_coarse_lines, int nout, const long long *map_dev,
                  int group, double scale, double *G_coarse, void *stream) {
    if (!G_fine || !map_dev || !G_coarse || group < 1 || nout < 1) return VP_EINVAL;
    const long long n = n_coarse_lines * nout;
    const double inv = (group & (group - 1)) == 0 ? 1.0 / group : 0.0;  // exact
    k_group_mean<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        G_fine, n, nout, make_fastdiv((unsigned)nout), map_dev, group, scale, inv, G_coarse);
    return cudaGetLastError() == cudaSuccess ? VP_OK : VP_ECUDA;
}

// Fine lines aggregated by every coarse line of a sweep, for a coarse grid
// whose velocity cells are factor^D fine cells (same spatial grid).
int vp_fluxnet_line_map(const vp_grid *fine, const vp_grid *coarse, int factor, int kick, int dim,
                        long long *map_host, long long *n_coarse_lines, int *group) {
    if (!fine || !coarse || factor < 1 || fine->dx != coarse->dx || fine->dx < 1 || fine->dx > 2) return VP_EINVAL;
    const int D = fine->dx;
    long long NXf = 1, NVf = 1, NVc = 1;
    for (int k = 0; k < D; ++k) {
        if (fine->nx[k] != coarse->nx[k] || fine->nv[k] != factor * coarse->nv[k]) return VP_EINVAL;
        NXf *= fine->nx[k];
        NVf *= fine->nv[k];
        NVc *= coarse->nv[k];
    }
    const LineGeo qc = line_geo(*coarse, NXf, NVc, kick, dim);
    const LineGeo qf = line_geo(*fine, NXf, NVf, kick, dim);
    const long long ncl = qc.outer * qc.inner;
    // velocity cells of the coarse line's other axes, expanded
    int g = 1;
    for (int k = 0; k < D; ++k)
        if (!(kick && k == dim)) g *= factor;
    if (n_coarse_lines) *n_coarse_lines = ncl;
    if (group) *group = g;
    if (!map_host) return VP_OK;
    for (long long cl = 0; cl < ncl; ++cl) {
        const long long O = cl / qc.inner, C = cl % qc.inner;
        // full coarse index of the line's first cell, decomposed [x..][J..]
        const long long lin = O * (long long)qc.L * qc.inner + C;
        long long x = lin / NVc, J = lin % NVc;
        int Jv[2] = {0, 0};
        for (int k = D - 1; k >= 0; --k) {
            Jv[k] = (int)(J % coarse->nv[k]);
            J /= coarse->nv[k];
        }
        int idx = 0;
        for (int a = 0; a < (D > 0 ? factor : 1); ++a)
            for (int b = 0; b < (D > 1 ? factor : 1); ++b) {
                int jf[2] = {Jv[0] * factor + a, D > 1 ? Jv[1] * factor + b : 0};
                // along the swept velocity axis every fine line starts at cell 0
                if (kick) {
                    if (dim == 0 && a) continue;
                    if (dim == 1 && b) continue;
                    jf[dim] = 0;
                }
                long long jl = 0;
                for (int k = 0; k < D; ++k) jl = jl * fine->nv[k] + jf[k];
                const long long flin = x * NVf + jl;  // fine index of the line's first cell
                const long long Of = flin / ((long long)qf.L * qf.inner);
                const long long Cf = flin % qf.inner;
                map_host[cl * g + idx++] = Of * qf.inner + Cf;
            }
    }
    return VP_OK;
}

int vp_make_samples(vp_ctx *coarse, int kick, int dim, double dt, const double *accel_dev,
                    const double *Gc_dev, double zmin, float *X_dev, float *y_dev, float *scale_dev) {
    vp_ctx *c = coarse;
    if (!c || !c->f || !Gc_dev || !X_dev || !y_dev) return VP_EINVAL;
    if (dim < 0 || dim >= c->g.dx || (kick && !accel_dev)) return vp_fail(c, VP_EINVAL, "bad sample arguments");
    const LineGeo q = line_geo(c->g, c->NX, c->NV, kick, dim);
    LineTile t = line_tile(q);
    int rc;
    if ((rc = vp_launch_shift_tables_f32(c, kick, 1u << dim, dt, accel_dev))) return rc;
    const LineShift<float> *tab = static_cast<const LineShift<float> *>(c->d_shift) + dim * c->shift_cap;
    const size_t xbytes = (size_t)kSampleThreads * NF * sizeof(float);
    auto bytes = [&](int W) { return xbytes + (size_t)3 * W * ((q.L + 2 * kEdge) | 1) * sizeof(float); };
    int W = 32;
    while (W > 1 && bytes(W) > 72 * 1024) W /= 2;  // three CTAs per SM
    const bool staged = bytes(W) <= 200 * 1024;
    set_width(t, staged ? W : 32);
    const unsigned blocks = (unsigned)((t.lines + t.W - 1) / t.W);
    const size_t smem = staged ? bytes(t.W) : xbytes;
    VP_CUDA_TRY(c, cudaFuncSetAttribute(k_make_samples<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    if (staged)
        k_make_samples<true><<<blocks, kSampleThreads, smem, c->stream>>>(
            static_cast<const float *>(c->f), t, tab, kick, accel_dev, q.lo, q.dvel, dt, q.h, Gc_dev, zmin, X_dev,
            y_dev, scale_dev, (float)c->g.alpha);
    else
        k_make_samples<false><<<blocks, kSampleThreads, smem, c->stream>>>(
            static_cast<const float *>(c->f), t, tab, kick, accel_dev, q.lo, q.dvel, dt, q.h, Gc_dev, zmin, X_dev,
            y_dev, scale_dev, (float)c->g.alpha);
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

}  // extern "C"

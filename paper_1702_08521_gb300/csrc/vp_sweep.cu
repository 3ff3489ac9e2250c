// vp_sweep.cu -- the SL-MPP5/7 advection sweep (shift decomposition, CSL
// flux, MP constraint, PP limiter, conservative update) for sm_103a.
//
// A sweep advances every 1D line of f along one phase-space axis.  f is seen
// as [outer][L][inner]: the line runs along the middle index with element
// stride `inner`.  Two kernels stage whole lines in shared memory so that
// every cell of f is read from HBM once and written once, in place:
//   * k_sweep_cols: inner > 1 (strided axes).  A CTA owns a tile of W
//     consecutive columns (W lines) x the full line; global loads and stores
//     are row-contiguous (coalesced, 16-byte vectors when aligned).
//   * k_sweep_rows: inner == 1 (the contiguous last velocity axis).  A CTA
//     owns R consecutive lines, one contiguous block of memory, staged with
//     an odd row pitch so that 32 lanes walking 32 lines hit 32 banks.
//   * k_sweep_cols_tma: the strided-axis sweep as a persistent kernel fed by
//     TMA: one elected thread streams [L x W] tiles global -> shared with
//     cp.async.bulk.tensor (two input stages, mbarrier completion), all
//     threads compute into a shared output tile, which TMA stores back while
//     the next tile is computed.  No per-thread global loads or stores.
// Each thread walks a segment of one line in the upwind direction with a
// sliding register window, so each interface flux is computed once and the
// incoming flux of a cell is the outgoing flux of its upwind neighbour.
#include <cudaTypedefs.h>

#include <cmath>

#include "vp_internal.cuh"
#include "vp_sweep_core.cuh"
#include "vp_tma.cuh"

// A translation unit holds the sweeps of one precision and order (the four
// compile in parallel): this file itself FP32 of order 7 and the dispatch, the
// files vp_sweep_*.cu that include it the others.
#ifndef VP_SWEEP_ORDER
#define VP_SWEEP_MAIN
#define VP_SWEEP_ORDER 7
#define VP_SWEEP_REAL float
#define VP_UNIT(name) name##_f32_o7
#endif
typedef VP_SWEEP_REAL unit_t;

namespace {

constexpr int kOrder = VP_SWEEP_ORDER;

using vp_core::line_class;
using vp_core::ShiftSrc;
using vp_core::walk;

// running-pointer store of one line's new values (element stride `step`
// between consecutive cells of the walk)
template <typename T>
struct PtrStore {
    T *p;
    long long step;
    __device__ __forceinline__ void operator()(int, T v) {
        *p = v;
        p += step;
    }
};

// staged-load strided sweep: tile = W columns x the whole line, staged as
// rows GP..GP+L-1 of a [(L + 2 GP)][W] shared tile; zero-inflow lines get GP =
// VP_GHOST zero rows on each side, periodic lines none.  PAIR (FP32 only): a
// thread walks two adjacent columns at once with the packed pair arithmetic
// (W / 2 threads per segment row); a pair whose lines differ in their integer
// shift or direction is walked one line after the other.
// largest CTA of the two-line kernels and the CTAs per SM their register
// budget must allow
#define VP_PAIR_THREADS 512
#define VP_PAIR_MINB 1

// GEN: any tile -- ragged last tiles, rows that are no multiple of 16 bytes,
// several narrow outer blocks side by side.  Not GEN: whole tiles of one block in
// 16-byte rows, a thread's rows at one column (the general tile's address
// arithmetic costs 3-6% there: Plummer 16^3 x 64^3 drift x1 1.86 against 1.97 ms).
template <typename T, int ORDER, bool PERIODIC, bool FULL, bool PAIR, bool FLAT, bool GEN>
__global__ void __launch_bounds__(PAIR ? VP_PAIR_THREADS : 512, PAIR ? VP_PAIR_MINB : 1)
    k_sweep_cols(T *f, const __grid_constant__ ShiftSrc<T> src, SweepGeo geo, LimParams lp) {
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr int GP = PERIODIC ? 0 : VP_GHOST;
    T *sm = reinterpret_cast<T *>(smraw);
    const int W = geo.W, L = geo.L;
    // W columns of one outer block, or (kblk > 1) kblk whole blocks side by side
    const bool packed = GEN && geo.kblk > 1;
    const unsigned o = packed ? blockIdx.x * (unsigned)geo.kblk : fdiv(blockIdx.x, geo.fd_tpo);
    const unsigned c0 = packed ? 0u : (blockIdx.x - o * geo.tpo) * (unsigned)W;
    const int nblk = packed ? (int)(geo.outer - o < geo.kblk ? geo.outer - o : geo.kblk) : 1;
    const int wc = !GEN ? W : (packed ? nblk * (int)geo.inner : (int)((geo.inner - c0) < W ? (geo.inner - c0) : W));
    T *const base0 = f + (long long)o * L * geo.inner + c0;
    // first cell of column cc, its outer block and inner index
    auto column = [&](int cc, unsigned &ob, unsigned &c) -> T * {
        const unsigned k = packed ? fdiv((unsigned)cc, geo.fd_inner) : 0u;
        ob = o + k;
        c = packed ? cc - k * (unsigned)geo.inner : c0 + cc;
        return packed ? base0 + (long long)k * L * geo.inner + c : base0 + cc;
    };
    T *data = sm + GP * W;  // row 0 of the line
    // the tile's shifts: its columns' classes (drift), or its spatial points (kick)
    unsigned q0 = 0;
    int ncl = 1;
    LineShift<T> *shifts = nullptr;
    const bool own_drift = !src.tab && !src.accel;  // shifts of the grid alone: nothing to wait for
    if (!own_drift) dep_wait();
    if (!src.tab) {
        shifts = reinterpret_cast<LineShift<T> *>(smraw + (((size_t)(L + 2 * GP) * W * sizeof(T) + 15) & ~size_t(15)));
        q0 = geo.cls_from_inner ? fdiv(c0, geo.fd_cdiv) : fdiv(o, geo.fd_cdiv);
        const unsigned q1 = geo.cls_from_inner ? fdiv(packed ? (unsigned)geo.inner - 1 : c0 + wc - 1, geo.fd_cdiv)
                                               : fdiv(o + nblk - 1, geo.fd_cdiv);
        ncl = (int)(q1 - q0) + 1;
        vp_core::tile_shifts(shifts, q0, ncl, src, geo);
    }
    if (own_drift) dep_wait();
    dep_launch();
    // Every piece of the tile in flight at once (cp.async), so the staging is not
    // limited by one outstanding load per thread: pieces of 16, 8 or 4 bytes, the
    // widest that the row stride and the tile width are multiples of.  A 22 x 20 x
    // 23 x 31 x 33 x 30 grid (rows of 8-byte pieces) staged by single loads took
    // 1.12-1.18 ms per sweep against 0.37 ms of HBM.
    if constexpr (!GEN) {
        constexpr int VEC = 16 / sizeof(T);
        const int wv = W / VEC;
        const int r = (int)fdiv(threadIdx.x, geo.fd_wv);
        const int cv = threadIdx.x - r * wv;
        const int rstep = (int)fdiv(blockDim.x, geo.fd_wv);
        const T *from = base0 + (long long)r * geo.inner + cv * VEC;
        T *dst = data + r * W + cv * VEC;
        const long long sstep = (long long)rstep * geo.inner;
        for (int rr = r; rr < L; rr += rstep) {
            vp_tma::cp_async16(dst, from);
            from += sstep;
            dst += rstep * W;
        }
    } else {
        const int wv = W / geo.vec;
        const int r = (int)fdiv(threadIdx.x, geo.fd_wv);
        const int cv = (threadIdx.x - r * wv) * geo.vec;
        const int rstep = (int)fdiv(blockDim.x, geo.fd_wv);
        if (r < rstep && cv < wc) {
            unsigned ob, c;
            const T *from = column(cv, ob, c) + (long long)r * geo.inner;
            T *dst = data + r * W + cv;
            const long long sstep = (long long)rstep * geo.inner;
            auto copy = [&](auto bytes) {
                for (int rr = r; rr < L; rr += rstep) {
                    vp_tma::cp_async<decltype(bytes)::value>(dst, from);
                    from += sstep;
                    dst += rstep * W;
                }
            };
            const int bytes = geo.vec * (int)sizeof(T);
            if (bytes == 16) copy(std::integral_constant<int, 16>());
            else if (bytes == 8) copy(std::integral_constant<int, 8>());
            else copy(std::integral_constant<int, 4>());
        }
    }
    // while the copies are under way: the zero rows, and the thread's column,
    // segment and shift
    for (int e = threadIdx.x; e < GP * W; e += blockDim.x) {
        sm[e] = T(0);
        data[L * W + e] = T(0);
    }
    const unsigned seg = fdiv(threadIdx.x, PAIR ? geo.fd_w2 : geo.fd_w);
    const int cc = PAIR ? 2 * (int)(threadIdx.x - seg * (unsigned)(W >> 1)) : (int)(threadIdx.x - seg * (unsigned)W);
    const bool act = cc < wc && (int)seg < geo.nseg;
    unsigned ob = 0, c = 0;
    T *const base = column(act ? cc : 0, ob, c);  // a pair's columns lie in one block (its width is even)
    LineShift<T> sa, sb;
    if (src.tab && act) {
        sa = src.tab[line_class(geo, ob, c)];
        if (PAIR) sb = src.tab[line_class(geo, ob, c + (cc + 1 < wc ? 1 : 0))];
    }
    vp_tma::cp_async_wait_all();
    __syncthreads();
    if (!src.tab) {
        vp_core::tile_weights(shifts, ncl, src);
        if (act) {
            sa = shifts[fdiv(geo.cls_from_inner ? c : ob, geo.fd_cdiv) - q0];
            if (PAIR) sb = shifts[fdiv(geo.cls_from_inner ? c + (cc + 1 < wc ? 1 : 0) : ob, geo.fd_cdiv) - q0];
        }
    }
    if (!act) return;
    constexpr int G1 = PERIODIC ? 1 : VP_GHOST;
    const int r0 = (int)fdiv(seg * (unsigned)L, geo.fd_nseg);
    const int r1 = (int)fdiv((seg + 1) * (unsigned)L, geo.fd_nseg);
    if constexpr (PAIR) {
        if (cc + 1 < wc) {
            if (sa.n == sb.n && sa.sigma == sb.sigma) {
                const vp_core::LineShiftP2 sh = vp_core::pair_shift(sa, sb);
                const int i0 = sh.sigma > 0 ? r0 : r1 - 1;
                PtrStore<vp_core::P2> st{reinterpret_cast<vp_core::P2 *>(base + (long long)i0 * geo.inner),
                                         (long long)sh.sigma * (geo.inner >> 1)};
                walk<vp_core::P2, ORDER, PERIODIC, FULL, G1, false, FLAT>(
                    reinterpret_cast<const vp_core::P2 *>(data + cc), W >> 1, L, sh, r0, r1,
                    vp_core::P2((float)lp.alpha), lp.mp, lp.pp, st);
                return;
            }
            const int i1 = sb.sigma > 0 ? r0 : r1 - 1;
            PtrStore<T> st{base + 1 + (long long)i1 * geo.inner, (long long)sb.sigma * geo.inner};
            walk<T, ORDER, PERIODIC, FULL, G1, false, FLAT>(data + cc + 1, W, L, sb, r0, r1, (T)lp.alpha, lp.mp,
                                                            lp.pp, st);
        }
        const int i0 = sa.sigma > 0 ? r0 : r1 - 1;
        PtrStore<T> st{base + (long long)i0 * geo.inner, (long long)sa.sigma * geo.inner};
        walk<T, ORDER, PERIODIC, FULL, G1, false, FLAT>(data + cc, W, L, sa, r0, r1, (T)lp.alpha, lp.mp, lp.pp, st);
    } else {
        const int i0 = sa.sigma > 0 ? r0 : r1 - 1;
        vp_core::walk_line<T, ORDER, PERIODIC, FULL, G1, FLAT>(
            data + cc, W, L, sa, r0, r1, (T)lp.alpha, lp.mp, lp.pp, [&](auto t) {
                using U = decltype(t);
                return PtrStore<U>{reinterpret_cast<U *>(base + (long long)i0 * geo.inner),
                                   (long long)sa.sigma * geo.inner};
            });
    }
}

// contiguous-axis sweep: R lines per CTA.  Input rows at odd pitch P with a
// zero ghost on each side, results to a second shared tile (odd pitch Q), then
// copied out with 16-byte coalesced stores.  PAIR (FP32 only): lines 2q and
// 2q + 1 are interleaved element by element in shared memory (pair pitch 2P,
// 2Q) so that one thread walks both with 8-byte loads and stores and the
// packed pair arithmetic; a pair whose lines differ in their integer shift or
// direction, and the odd last line of a ragged tile, are walked one line at
// a time (element stride 2).  The 16-lane phases of 8-byte accesses stay
// conflict-free because P is odd.
template <typename T, int ORDER, bool PERIODIC, bool FULL, bool PAIR, bool FLAT>
__global__ void __launch_bounds__(PAIR ? VP_PAIR_THREADS : 512, PAIR ? VP_PAIR_MINB : 1)
    k_sweep_rows(T *f, const __grid_constant__ ShiftSrc<T> src, SweepGeo geo, LimParams lp) {
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr int GP = PERIODIC ? 0 : VP_GHOST;
    const int L = geo.L, R = geo.R;
    const int P = (L + 2 * GP) | 1;
    const int Q = L | 1;
    T *in = reinterpret_cast<T *>(smraw);
    T *out = in + R * P;
    const long long l0 = (long long)blockIdx.x * R;
    const int nl = (int)((geo.outer - l0) < R ? (geo.outer - l0) : R);
    T *base = f + l0 * L;
    const int tot = nl * L;
    // the tile's shifts: a kick's lines belong to consecutive spatial points
    // (drifts along contiguous lines, one velocity cell, read the table)
    unsigned q0 = 0;
    int ncl = 1;
    LineShift<T> *shifts = nullptr;
    dep_wait();
    dep_launch();
    if (!src.tab) {
        shifts = reinterpret_cast<LineShift<T> *>(smraw + (((size_t)R * (P + Q) * sizeof(T) + 15) & ~size_t(15)));
        q0 = fdiv((unsigned)l0, geo.fd_cdiv);
        ncl = (int)(fdiv((unsigned)(l0 + nl - 1), geo.fd_cdiv) - q0) + 1;
        vp_core::tile_shifts(shifts, q0, ncl, src, geo);
    }
    auto shift_of = [&](int line) -> LineShift<T> {
        if (src.tab) return src.tab[line_class(geo, (unsigned)(l0 + line), 0u)];
        return shifts[fdiv((unsigned)(l0 + line), geo.fd_cdiv) - q0];
    };
    // shared-memory index of cell pos of line r in the input / output tile
    auto iidx = [&](int r, int pos) -> int {
        return PAIR ? (r >> 1) * (2 * P) + 2 * (GP + pos) + (r & 1) : r * P + GP + pos;
    };
    auto oidx = [&](int r, int pos) -> int { return PAIR ? (r >> 1) * (2 * Q) + 2 * pos + (r & 1) : r * Q + pos; };
    if (GP > 0) {
        constexpr int G = GP > 0 ? GP : 1;
        for (int e = threadIdx.x; e < nl * G; e += blockDim.x) {
            const int r = e / G, k = e - r * G;
            in[iidx(r, k - G)] = T(0);
            in[iidx(r, L + k)] = T(0);
        }
    }
    constexpr int VEC = 16 / sizeof(T);
    const bool vec = (L % VEC) == 0;
    // lines whose length is no multiple of a 16-byte piece: the tile is still one
    // run of memory, and a piece's elements fall into at most two lines
    const bool ragged = !vec && L >= VEC && (reinterpret_cast<uintptr_t>(base) & 15) == 0;
    constexpr int ES = PAIR ? 2 : 1;  // shared-memory stride between a line's cells
    // Element e = r L + pos of the tile: a thread starts at e = VEC t (or t)
    // and advances by a fixed (rows, positions) step, so no division per element.
    if (vec) {
        // 16-byte loads in flight per thread (Plummer 16^3 x 64^3 contiguous kick:
        // 2 loads 2.20 ms, 4 2.10, 8 2.04; cell-by-cell cp.async, without the bank
        // conflicts of these stores, 3.16: the copies' instruction rate counts)
        constexpr int U = 8;
        const int st = blockDim.x * VEC;
        const int dr = (int)fdiv(st, geo.fd_l), dp = st - dr * L;
        int r = (int)fdiv(threadIdx.x * VEC, geo.fd_l), pos = threadIdx.x * VEC - r * L;
        int e = threadIdx.x * VEC;
        for (; e + (U - 1) * st < tot; e += U * st) {
            float4 x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = *reinterpret_cast<const float4 *>(base + e + u * st);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const T *xv = reinterpret_cast<const T *>(&x[u]);
                const int i0 = iidx(r, pos);
#pragma unroll
                for (int k = 0; k < VEC; ++k) in[i0 + (PAIR ? 2 * k : k)] = xv[k];
                r += dr;
                pos += dp;
                if (pos >= L) {
                    pos -= L;
                    ++r;
                }
            }
        }
        for (; e < tot; e += st) {
            const float4 x = *reinterpret_cast<const float4 *>(base + e);
            const T *xv = reinterpret_cast<const T *>(&x);
            const int i0 = iidx(r, pos);
#pragma unroll
            for (int k = 0; k < VEC; ++k) in[i0 + (PAIR ? 2 * k : k)] = xv[k];
            r += dr;
            pos += dp;
            if (pos >= L) {
                pos -= L;
                ++r;
            }
        }
    } else if (ragged) {
        constexpr int U = 8;  // 16-byte loads in flight per thread
        const int st = blockDim.x * VEC;
        const int dr = (int)fdiv(st, geo.fd_l), dp = st - dr * L;
        int r = (int)fdiv(threadIdx.x * VEC, geo.fd_l), pos = threadIdx.x * VEC - r * L;
        const int whole = tot - tot % VEC;
        for (int e = threadIdx.x * VEC; e < whole; e += U * st) {
            float4 x[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (e + u * st < whole) x[u] = *reinterpret_cast<const float4 *>(base + e + u * st);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (e + u * st >= whole) break;
                const T *xv = reinterpret_cast<const T *>(&x[u]);
                const int i0 = iidx(r, pos), i1 = iidx(r + 1, pos - L);
#pragma unroll
                for (int k = 0; k < VEC; ++k) in[(pos + k < L ? i0 : i1) + ES * k] = xv[k];
                r += dr;
                pos += dp;
                if (pos >= L) {
                    pos -= L;
                    ++r;
                }
            }
        }
        for (int e = whole + threadIdx.x; e < tot; e += blockDim.x) in[iidx(nl - 1, e - (nl - 1) * L)] = base[e];
    } else {
        const int dr = (int)fdiv(blockDim.x, geo.fd_l), dp = blockDim.x - dr * L;
        int r = (int)fdiv(threadIdx.x, geo.fd_l), pos = threadIdx.x - r * L;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            in[iidx(r, pos)] = base[e];
            r += dr;
            pos += dp;
            if (pos >= L) {
                pos -= L;
                ++r;
            }
        }
    }
    __syncthreads();
    if (!src.tab) vp_core::tile_weights(shifts, ncl, src);
    constexpr int G1 = PERIODIC ? 1 : VP_GHOST;
    if constexpr (PAIR) {
        const unsigned seg = fdiv(threadIdx.x, geo.fd_w2);
        const int line = 2 * (int)(threadIdx.x - seg * (unsigned)(R >> 1));
        if (line < nl && (int)seg < geo.nseg) {
            const int r0 = (int)fdiv(seg * (unsigned)L, geo.fd_nseg);
            const int r1 = (int)fdiv((seg + 1) * (unsigned)L, geo.fd_nseg);
            const LineShift<float> sa = shift_of(line);
            bool paired = false;
            if (line + 1 < nl) {
                const LineShift<float> sb = shift_of(line + 1);
                if (sa.n == sb.n && sa.sigma == sb.sigma) {
                    const vp_core::LineShiftP2 sh = vp_core::pair_shift(sa, sb);
                    const int i0 = sh.sigma > 0 ? r0 : r1 - 1;
                    PtrStore<vp_core::P2> st{reinterpret_cast<vp_core::P2 *>(out + oidx(line, i0)), sh.sigma};
                    walk<vp_core::P2, ORDER, PERIODIC, FULL, G1, false, FLAT>(
                        reinterpret_cast<const vp_core::P2 *>(in + iidx(line, 0)), 1, L, sh, r0, r1,
                        vp_core::P2((float)lp.alpha), lp.mp, lp.pp, st);
                    paired = true;
                } else {
                    const int i1 = sb.sigma > 0 ? r0 : r1 - 1;
                    PtrStore<T> st{out + oidx(line + 1, i1), 2LL * sb.sigma};
                    walk<T, ORDER, PERIODIC, FULL, G1, false, FLAT>(in + iidx(line + 1, 0), 2, L, sb, r0, r1, (T)lp.alpha,
                                                       lp.mp, lp.pp, st);
                }
            }
            if (!paired) {
                const int i0 = sa.sigma > 0 ? r0 : r1 - 1;
                PtrStore<T> st{out + oidx(line, i0), 2LL * sa.sigma};
                walk<T, ORDER, PERIODIC, FULL, G1, false, FLAT>(in + iidx(line, 0), 2, L, sa, r0, r1, (T)lp.alpha, lp.mp,
                                                   lp.pp, st);
            }
        }
    } else {
        const unsigned seg = fdiv(threadIdx.x, geo.fd_w);
        const int line = (int)(threadIdx.x - seg * (unsigned)R);
        if (line < nl && (int)seg < geo.nseg) {
            const LineShift<T> sh = shift_of(line);
            const int r0 = (int)fdiv(seg * (unsigned)L, geo.fd_nseg);
            const int r1 = (int)fdiv((seg + 1) * (unsigned)L, geo.fd_nseg);
            const int i0 = sh.sigma > 0 ? r0 : r1 - 1;
            vp_core::walk_line<T, ORDER, PERIODIC, FULL, G1, FLAT>(
                in + line * P + GP, 1, L, sh, r0, r1, (T)lp.alpha, lp.mp, lp.pp, [&](auto t) {
                    using U = decltype(t);
                    return PtrStore<U>{reinterpret_cast<U *>(out + line * Q + i0), (long long)sh.sigma};
                });
        }
    }
    __syncthreads();
    if (vec) {
        const int st = blockDim.x * VEC;
        const int dr = (int)fdiv(st, geo.fd_l), dp = st - dr * L;
        int r = (int)fdiv(threadIdx.x * VEC, geo.fd_l), pos = threadIdx.x * VEC - r * L;
        for (int e = threadIdx.x * VEC; e < tot; e += st) {
            float4 x;
            T *xv = reinterpret_cast<T *>(&x);
            const int o0 = oidx(r, pos);
#pragma unroll
            for (int k = 0; k < VEC; ++k) xv[k] = out[o0 + (PAIR ? 2 * k : k)];
            *reinterpret_cast<float4 *>(base + e) = x;
            r += dr;
            pos += dp;
            if (pos >= L) {
                pos -= L;
                ++r;
            }
        }
    } else if (ragged) {
        const int st = blockDim.x * VEC;
        const int dr = (int)fdiv(st, geo.fd_l), dp = st - dr * L;
        int r = (int)fdiv(threadIdx.x * VEC, geo.fd_l), pos = threadIdx.x * VEC - r * L;
        const int whole = tot - tot % VEC;
        for (int e = threadIdx.x * VEC; e < whole; e += st) {
            float4 x;
            T *xv = reinterpret_cast<T *>(&x);
            const int o0 = oidx(r, pos), o1 = oidx(r + 1, pos - L);
#pragma unroll
            for (int k = 0; k < VEC; ++k) xv[k] = out[(pos + k < L ? o0 : o1) + ES * k];
            *reinterpret_cast<float4 *>(base + e) = x;
            r += dr;
            pos += dp;
            if (pos >= L) {
                pos -= L;
                ++r;
            }
        }
        for (int e = whole + threadIdx.x; e < tot; e += blockDim.x) base[e] = out[oidx(nl - 1, e - (nl - 1) * L)];
    } else {
        const int dr = (int)fdiv(blockDim.x, geo.fd_l), dp = blockDim.x - dr * L;
        int r = (int)fdiv(threadIdx.x, geo.fd_l), pos = threadIdx.x - r * L;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            base[e] = out[oidx(r, pos)];
            r += dr;
            pos += dp;
            if (pos >= L) {
                pos -= L;
                ++r;
            }
        }
    }
}

// TMA-fed persistent strided sweep (two input and two output stages)
template <typename T, int ORDER, bool PERIODIC, bool FULL>
__global__ void __launch_bounds__(512) k_sweep_cols_tma(const __grid_constant__ CUtensorMap tmap,
                                                        const LineShift<T> *__restrict__ tab,
                                                        SweepGeo geo, LimParams lp,
                                                        int *__restrict__ status, unsigned wait_limit) {
    extern __shared__ __align__(128) unsigned char smraw_tma[];
    unsigned char *smraw = smraw_tma;
    __shared__ __align__(8) uint64_t bar[2];
    constexpr int GP = PERIODIC ? 0 : VP_GHOST;
    const int W = geo.W, L = geo.L;
    const int itile = (L + 2 * GP) * W;  // input stage: GP zero rows, L rows, GP zero rows
    const int otile = L * W;
    // TMA tensor copies need 128-byte aligned shared-memory buffers: align
    // the dynamic region explicitly (the launch reserves 128 spare bytes)
    const uint32_t sbase = vp_tma::saddr(smraw);
    const uint32_t pad = (128u - (sbase & 127u)) & 127u;
    T *in_buf = reinterpret_cast<T *>(smraw + pad);  // [2][L + 2 GP][W]
    T *out_buf = in_buf + 2 * itile;                  // [2][L][W]
    const unsigned tpo = geo.tpo;
    const unsigned ntiles = (unsigned)geo.outer * tpo;
    const uint32_t bytes = (uint32_t)(otile * sizeof(T));
    // self-check of every alignment the copies rely on; on failure report and
    // leave before issuing any copy
    if (((vp_tma::saddr(in_buf + GP * W) | vp_tma::saddr(in_buf + itile + GP * W) | vp_tma::saddr(out_buf) |
          vp_tma::saddr(out_buf + otile)) & 127u) != 0 ||
        ((W * sizeof(T)) & 127u) != 0) {
        if (threadIdx.x == 0) atomicExch(status, VP_EINVAL);
        return;
    }
    for (int e = threadIdx.x; e < GP * W; e += blockDim.x) {
        in_buf[e] = T(0);
        in_buf[(GP + L) * W + e] = T(0);
        in_buf[itile + e] = T(0);
        in_buf[itile + (GP + L) * W + e] = T(0);
    }
    if (threadIdx.x == 0) {
        vp_tma::mbar_init(&bar[0], 1);
        vp_tma::mbar_init(&bar[1], 1);
        vp_tma::fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            const unsigned t = blockIdx.x + (unsigned)s * gridDim.x;
            if (t < ntiles) {
                vp_tma::mbar_expect_tx(&bar[s], bytes);
                vp_tma::load_3d(in_buf + s * itile + GP * W, &tmap, &bar[s], (int)((t % tpo) * W), 0,
                                (int)(t / tpo));
            }
        }
    }
    const unsigned seg = fdiv(threadIdx.x, geo.fd_w);
    const int cc = (int)(threadIdx.x - seg * (unsigned)W);
    const int r0 = (int)fdiv(seg * (unsigned)L, geo.fd_nseg);
    const int r1 = (int)fdiv((seg + 1) * (unsigned)L, geo.fd_nseg);
    int k = 0;
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x, ++k) {
        const int s = k & 1;
        T *in = in_buf + s * itile;
        T *out = out_buf + s * otile;
        const bool arrived = vp_tma::mbar_wait(&bar[s], (uint32_t)((k >> 1) & 1), wait_limit);
        if (__syncthreads_or(!arrived)) {
            // a thread gave up on the tile: report, wait (bounded) for this
            // CTA's loads still in flight (this tile's and the next one's)
            // and for its stores, leave
            if (threadIdx.x == 0) {
                atomicExch(status, VP_ETIMEOUT);
                vp_tma::mbar_wait(&bar[s], (uint32_t)((k >> 1) & 1), 1u << 22);
                if (t + gridDim.x < ntiles) vp_tma::mbar_wait(&bar[s ^ 1], (uint32_t)(((k + 1) >> 1) & 1), 1u << 22);
                vp_tma::wait_all<0>();
            }
            return;
        }
        const unsigned o = fdiv(t, geo.fd_tpo);
        const unsigned c0 = (t - o * tpo) * (unsigned)W;
        const int wc = (int)((geo.inner - c0) < W ? (geo.inner - c0) : W);
        if (cc < wc && (int)seg < geo.nseg) {
            const LineShift<T> sh = tab[line_class(geo, o, c0 + cc)];
            const int i0 = sh.sigma > 0 ? r0 : r1 - 1;
            PtrStore<T> st{out + cc + i0 * W, (long long)sh.sigma * W};
            walk<T, ORDER, PERIODIC, FULL, PERIODIC ? 1 : VP_GHOST>(in + GP * W + cc, W, L, sh, r0, r1,
                                                                     (T)lp.alpha, lp.mp, lp.pp, st);
        }
        vp_tma::fence_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) {
            vp_tma::store_3d(&tmap, out, (int)c0, 0, (int)o);
            vp_tma::commit();
            const unsigned tn = t + 2u * gridDim.x;
            if (tn < ntiles) {
                vp_tma::mbar_expect_tx(&bar[s], bytes);
                const unsigned on = fdiv(tn, geo.fd_tpo);
                vp_tma::load_3d(in + GP * W, &tmap, &bar[s], (int)((tn - on * tpo) * W), 0, (int)on);
            }
            vp_tma::wait_read<1>();  // the other output tile is free again
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) vp_tma::wait_all<0>();
}

// Shift decomposition of every line class of the sweeps along the axes
// `dims` (one table per axis, `cap` entries apart), in double precision so that
// the integer part is exact: s = c dt / h, n = nearest integer (halves away from
// zero), zeta = s - n, nu = |zeta|; the weights are the CSL polynomials at nu.
// Eight lanes per class, one weight each (one thread per class spent 5.5 us in a
// chain of 49 FP64 FMAs and a division), and the axes of a stage in one launch.
struct TableAxes {
    int n;
    int dim[3], nclass[3];
    double lo[3], dvel[3], h[3];
    const double *accel[3];
};

template <typename T>
__global__ void k_shift_table(LineShift<T> *tab, long long cap, int kick, const __grid_constant__ TableAxes ax,
                              double dt, const __grid_constant__ WPoly wp) {
    dep_wait();
    dep_launch();
    const int a = blockIdx.y;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (int)(t >> 3), k = (int)t & 7;
    if ((t >> 3) >= ax.nclass[a]) return;
    LineShift<T> *e = tab + ax.dim[a] * cap + c;
    const double speed = kick ? ax.accel[a][c] : vp_core::cell_centre(ax.lo[a], ax.dvel[a], c);
    LineShift<T> sh;
    const double nu = vp_core::split_shift(speed, dt, ax.h[a], sh);
    if (k < 7) {
        e->w[k] = (T)vp_core::csl_weight(wp, k, nu);
    } else {
        e->nu = sh.nu;
        e->n = sh.n;
        e->sigma = sh.sigma;
    }
}

// a staged tile of at most 200 KB and up to 128 shifts behind it
constexpr int kSweepSmem = 216 * 1024;

template <typename T, int ORDER, bool PER, bool FULL, bool PAIR>
void set_attrs_pair() {
    constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaFuncSetAttribute(k_sweep_cols<T, ORDER, PER, FULL, PAIR, true, false>, attr, kSweepSmem);
    cudaFuncSetAttribute(k_sweep_cols<T, ORDER, PER, FULL, PAIR, !FULL, false>, attr, kSweepSmem);
    cudaFuncSetAttribute(k_sweep_cols<T, ORDER, PER, FULL, PAIR, true, true>, attr, kSweepSmem);
    cudaFuncSetAttribute(k_sweep_rows<T, ORDER, PER, FULL, PAIR, true>, attr, kSweepSmem);
    cudaFuncSetAttribute(k_sweep_rows<T, ORDER, PER, FULL, PAIR, !FULL>, attr, kSweepSmem);
}

template <typename T, int ORDER, bool PER, bool FULL>
void set_attrs_one() {
    set_attrs_pair<T, ORDER, PER, FULL, false>();
    if constexpr (sizeof(T) == 4) set_attrs_pair<T, ORDER, PER, FULL, true>();
    cudaFuncSetAttribute(k_sweep_cols_tma<T, ORDER, PER, FULL>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
}

template <typename T>
void set_attrs() {
    set_attrs_one<T, kOrder, true, true>();
    set_attrs_one<T, kOrder, false, true>();
    set_attrs_one<T, kOrder, true, false>();
    set_attrs_one<T, kOrder, false, false>();
}

// compile-time dispatch on the line's periodicity and whether both limiters
// are on (the scheme's order is the unit's)
#define VP_DISPATCH(PER_, FULL_, CALL)                 \
    do {                                               \
        if (PER_) {                                    \
            if (FULL_) { CALL(kOrder, true, true); }   \
            else { CALL(kOrder, true, false); }        \
        } else {                                       \
            if (FULL_) { CALL(kOrder, false, true); }  \
            else { CALL(kOrder, false, false); }       \
        }                                              \
    } while (0)

// geometry of the sweep along axis `dim` (kick: velocity axis, else spatial)

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        cudaGetLastError();
    }
    return fn;
}

// one sweep's speeds: class c of a kick moves at accel[c]; tab_ready: the
// context's table already holds this sweep's shifts, from class cls0 on
struct SweepShift {
    int kick, dim;
    double dt;
    const double *accel;
    bool tab_ready;
    long long cls0;
};

// ghost rows staged on each side of a line
inline int ghost_rows(const SweepGeo &geo) { return geo.periodic ? 0 : VP_GHOST; }

template <typename T>
size_t tma_smem(int L, int W, int gp) {
    return (size_t)(2 * (L + 2 * gp) * W + 2 * L * W) * sizeof(T) + 128;
}

template <typename T>
bool tma_eligible(const vp_ctx *c, const SweepGeo &geo, int W) {
    constexpr int VEC = 16 / sizeof(T);
    return geo.inner > 1 && geo.inner % VEC == 0 && W % VEC == 0 && geo.inner < (1LL << 31) &&
           geo.outer < (1LL << 31) && geo.L <= 256 && W <= 256 &&
           (W * sizeof(T)) % 128 == 0 && tma_smem<T>(geo.L, W, ghost_rows(geo)) <= 200 * 1024 &&
           tensor_map_encoder() != nullptr &&
           (reinterpret_cast<uintptr_t>(c->f) & 15) == 0;
}

// the pair walker: FP32, even columns per tile and row stride (8-byte pairs)
template <typename T>
bool pair_eligible(const vp_ctx *c, const SweepGeo &geo, int W) {
    return sizeof(T) == 4 && geo.inner > 1 && geo.inner % 2 == 0 && W % 2 == 0 &&
           (reinterpret_cast<uintptr_t>(c->f) & 7) == 0;
}

// line classes and tile coordinates are computed in 32-bit arithmetic
inline bool geo_fits_32(const SweepGeo &geo) { return geo.outer < (1LL << 32) && geo.inner < (1LL << 32); }

// The most classes a tile of w columns (or lines) meets, and whether its CTAs
// decompose their own shifts (true) or read a table that a launch of its own
// makes first.  Own shifts pay while the whole sweep is at most four CTAs per
// SM: the table's launch and the wait for it cost 3-4 us there, the FP64 chain
// in front of the walk well under 1 us.  With more waves the chain is paid by
// every wave (kicks of the 32^3 x 64^3 grid, one class per tile: 109 -> 119 ms
// per step), the table once.
inline int tile_classes(const SweepGeo &geo, int w) {
    const bool many = geo.cls_from_inner || geo.inner == 1;
    const long long n = many ? (w - 1) / geo.cdiv + 2 : (geo.kblk > 1 ? (geo.kblk - 1) / geo.cdiv + 2 : 1);
    return (int)(n > w ? w : n);
}
inline bool own_shifts(const vp_ctx *c, const SweepGeo &geo, long long tiles) {
    return !(geo.cls_from_inner && geo.inner == 1) && tiles <= 4LL * c->sm_count;
}

// the tile's shift source: own (ncl > 0) or the context's table, made here
template <typename T>
int shift_source(vp_ctx *c, const SweepShift &sw, const SweepGeo &geo, int w, long long tiles, bool table,
                 ShiftSrc<T> &src) {
    const vp_grid &g = c->g;
    src = ShiftSrc<T>{};
    if (!table && !sw.tab_ready && own_shifts(c, geo, tiles)) {
        const int d = sw.dim;
        src.accel = sw.kick ? sw.accel : nullptr;
        src.lo = g.vlo[d];
        src.dvel = (g.vhi[d] - g.vlo[d]) / g.nv[d];
        src.h = sw.kick ? src.dvel : (g.xhi[d] - g.xlo[d]) / g.nx[d];
        src.dt = sw.dt;
        src.ncl = tile_classes(geo, w);
        src.wp = c->wp;
        return VP_OK;
    }
    src.tab = static_cast<const LineShift<T> *>(c->d_shift) + sw.dim * c->shift_cap;
    if (sw.tab_ready) {
        src.tab += sw.cls0;
        return VP_OK;
    }
    return vp_launch_shift_tables(c, sw.kick, 1u << sw.dim, sw.dt, sw.accel);
}

template <typename T>
int launch_cols(vp_ctx *c, SweepGeo geo, const SweepTune &tu, const SweepShift &sw) {
    if (!geo_fits_32(geo)) return vp_fail(c, VP_ENOTSUP, "sweep geometry exceeds 32-bit line indexing");
    const LimParams lp{c->g.alpha, c->g.mp, c->g.pp};
    T *f = static_cast<T *>(c->f);
    const int L = geo.L;
    int W = tu.W;
    geo.kblk = 1;
    if (geo.inner < W) {
        // narrow blocks: as many whole ones side by side as the tile holds (30
        // columns of 33 cells, one block per CTA: 1.18 ms, a warp of them idle)
        const int wt = (int)geo.inner;
        const bool tma = tu.impl == 2 && tma_eligible<T>(c, geo, wt);
        long long k = tma ? 1 : W / wt;
        // (of lines so long that W columns do not fit, as many as do)
        const long long fit = 200 * 1024 / ((long long)(L + 2 * ghost_rows(geo)) * wt * (int)sizeof(T));
        k = k > fit && fit > 0 ? fit : k;
        k = k > geo.outer ? geo.outer : k;
        geo.kblk = (int)k;
        W = wt * geo.kblk;
    }
    const bool pair = tu.impl == 3 && pair_eligible<T>(c, geo, W);
    // walkers per segment row: W lines, or W / 2 line pairs; at most 512 threads
    const int per_row = pair ? W >> 1 : W;
    int nseg = tu.nseg;
    while (nseg > 1 && per_row * nseg > (pair ? VP_PAIR_THREADS : 512)) nseg >>= 1;
    geo.W = W;
    geo.nseg = nseg;
    // the widest pieces the rows are made of
    geo.vec = 16 / (int)sizeof(T);
    while (geo.inner % geo.vec || W % geo.vec) geo.vec /= 2;
    const int wv = W / geo.vec;
    int threads = ((per_row * nseg + 31) / 32) * 32;
    if (threads < wv) threads = (wv + 31) / 32 * 32;  // one row of pieces at least
    const long long tiles = geo.kblk > 1 ? (geo.outer + geo.kblk - 1) / geo.kblk
                                         : geo.outer * ((geo.inner + W - 1) / W);
    if (tiles >= (1LL << 31)) return vp_fail(c, VP_ENOTSUP, "sweep has too many tiles");
    geo.tpo = (unsigned)((geo.inner + W - 1) / W);
    geo.fd_tpo = make_fastdiv(geo.tpo);
    geo.fd_w = make_fastdiv((unsigned)W);
    geo.fd_nseg = make_fastdiv((unsigned)nseg);
    geo.fd_wv = make_fastdiv((unsigned)wv);
    geo.fd_inner = make_fastdiv((unsigned)geo.inner);
    const bool per = geo.periodic != 0;
    const bool full = c->g.mp && c->g.pp;
    const bool flat = tu.flat;
    const bool tma = tu.impl == 2 && tma_eligible<T>(c, geo, W);
    const size_t tile = (size_t)(L + 2 * ghost_rows(geo)) * W * sizeof(T);
    if (!tma && tile > 200 * 1024) return vp_fail(c, VP_ENOTSUP, "line of %d cells too long to stage", L);
    ShiftSrc<T> src;
    const int rc = shift_source<T>(c, sw, geo, W, tiles, tma, src);
    if (rc) return rc;
    const size_t smem = tile + vp_core::shift_smem<T>(tile, src.ncl);
    if (tma) {
        const LineShift<T> *tab = src.tab;
        CUtensorMap map;
        const cuuint64_t dims[3] = {(cuuint64_t)geo.inner, (cuuint64_t)L, (cuuint64_t)geo.outer};
        const cuuint64_t strides[2] = {(cuuint64_t)geo.inner * sizeof(T),
                                       (cuuint64_t)geo.inner * L * sizeof(T)};
        const cuuint32_t box[3] = {(cuuint32_t)W, (cuuint32_t)L, 1};
        const cuuint32_t estr[3] = {1, 1, 1};
        CUresult r = tensor_map_encoder()(&map, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                                               : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                                          3, f, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return vp_fail(c, VP_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
        const size_t tsmem = tma_smem<T>(L, W, ghost_rows(geo));
        int per_sm = tu.ctas_per_sm;
        if (per_sm <= 0) {
#define VP_OCC(O, P, F) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep_cols_tma<T, O, P, F>, threads, tsmem)
            VP_DISPATCH(per, full, VP_OCC);
#undef VP_OCC
            per_sm = per_sm < 1 ? 1 : per_sm;
        }
        long long grid = (long long)per_sm * c->sm_count;
        grid = grid > tiles ? tiles : grid;
#define VP_LAUNCH(O, P, F) \
    k_sweep_cols_tma<T, O, P, F><<<(unsigned)grid, threads, tsmem, c->stream>>>(map, tab, geo, lp, c->d_status, \
                                                                                c->opt_wait_limit)
        VP_DISPATCH(per, full, VP_LAUNCH);
#undef VP_LAUNCH
    } else {
        geo.fd_w2 = make_fastdiv((unsigned)(W >> 1 > 0 ? W >> 1 : 1));
        const bool gen = geo.kblk > 1 || geo.vec * sizeof(T) != 16 || geo.inner % W || threads % wv;
#define VP_LAUNCH_COLS(O, P, F, PAIR)                                                                              \
    if (gen)                                                                                                       \
        vp_launch_dep(k_sweep_cols<T, O, P, F, PAIR, true, true>, (unsigned)tiles, threads, smem, c->stream, f, \
                      src, geo, lp); \
    else if (flat)                                                                                                 \
        vp_launch_dep(k_sweep_cols<T, O, P, F, PAIR, true, false>, (unsigned)tiles, threads, smem, c->stream, f, \
                      src, geo, lp); \
    else                                                                                                           \
        vp_launch_dep(k_sweep_cols<T, O, P, F, PAIR, !F, false>, (unsigned)tiles, threads, smem, c->stream, f, \
                      src, geo, lp)
#define VP_LAUNCH(O, P, F)                          \
    if (pair) {                                     \
        VP_LAUNCH_COLS(O, P, F, sizeof(T) == 4);    \
    } else {                                        \
        VP_LAUNCH_COLS(O, P, F, false);             \
    }
        VP_DISPATCH(per, full, VP_LAUNCH);
#undef VP_LAUNCH
#undef VP_LAUNCH_COLS
    }
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

template <typename T>
size_t rows_smem(int L, int R, int gp) {
    return (size_t)R * (((L + 2 * gp) | 1) + (L | 1)) * sizeof(T);
}

template <typename T>
int launch_rows(vp_ctx *c, SweepGeo geo, const SweepTune &tu, const SweepShift &sw) {
    if (!geo_fits_32(geo)) return vp_fail(c, VP_ENOTSUP, "sweep geometry exceeds 32-bit line indexing");
    const LimParams lp{c->g.alpha, c->g.mp, c->g.pp};
    T *f = static_cast<T *>(c->f);
    const int L = geo.L;
    int R = tu.W;
    if (geo.outer < R) R = (int)geo.outer;
    const bool pair = tu.impl == 3 && sizeof(T) == 4;
    if (pair && (R & 1)) ++R;  // a single ragged tile keeps an empty slot
    // walkers per segment row: R lines, or R / 2 line pairs; at most 512 threads
    const int per_row = pair ? R >> 1 : R;
    int nseg = tu.nseg;
    while (nseg > 1 && per_row * nseg > (pair ? VP_PAIR_THREADS : 512)) nseg >>= 1;
    geo.R = R;
    geo.nseg = nseg;
    geo.fd_w = make_fastdiv((unsigned)R);
    geo.fd_nseg = make_fastdiv((unsigned)nseg);
    geo.fd_l = make_fastdiv((unsigned)L);
    const long long blocks = (geo.outer + R - 1) / R;
    if (blocks >= (1LL << 31)) return vp_fail(c, VP_ENOTSUP, "sweep has too many tiles");
    const size_t tile = rows_smem<T>(L, R, ghost_rows(geo));
    if (tile > 200 * 1024) return vp_fail(c, VP_ENOTSUP, "line of %d cells too long to stage", L);
    ShiftSrc<T> src;
    const int rc = shift_source<T>(c, sw, geo, R, blocks, false, src);
    if (rc) return rc;
    const size_t smem = tile + vp_core::shift_smem<T>(tile, src.ncl);
    const int threads = ((per_row * nseg + 31) / 32) * 32;
    const bool per = geo.periodic != 0;
    const bool full = c->g.mp && c->g.pp;
    const bool flat = tu.flat;
    if (pair) {
        geo.fd_w2 = make_fastdiv((unsigned)(R >> 1));
        const int pthreads = threads;
#define VP_LAUNCH(O, P, F)                                                                                     \
    if (flat)                                                                                                  \
        vp_launch_dep(k_sweep_rows<T, O, P, F, sizeof(T) == 4, true>, (unsigned)blocks, pthreads, smem, \
                      c->stream, f, src, geo, lp); \
    else                                                                                                       \
        vp_launch_dep(k_sweep_rows<T, O, P, F, sizeof(T) == 4, !F>, (unsigned)blocks, pthreads, smem, c->stream, \
                      f, src, geo, lp)
        VP_DISPATCH(per, full, VP_LAUNCH);
#undef VP_LAUNCH
    } else {
#define VP_LAUNCH(O, P, F)                                                                                     \
    if (flat)                                                                                                  \
        vp_launch_dep(k_sweep_rows<T, O, P, F, false, true>, (unsigned)blocks, threads, smem, c->stream, f, src, \
                      geo, lp); \
    else                                                                                                       \
        vp_launch_dep(k_sweep_rows<T, O, P, F, false, !F>, (unsigned)blocks, threads, smem, c->stream, f, src, \
                      geo, lp)
        VP_DISPATCH(per, full, VP_LAUNCH);
#undef VP_LAUNCH
    }
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

// default tile choice when the autotuner has not run
template <typename T>
SweepTune default_tune(const vp_ctx *c, const SweepGeo &geo) {
    SweepTune tu{};
    tu.valid = 1;
    tu.flat = 1;
    const int L = geo.L;
    if (geo.inner > 1) {
        int W = (int)(32768 / sizeof(T) / L);  // ~32 KB staged tile
        W = W > 128 ? 128 : (W < 32 ? 32 : W);
        W &= ~3;
        // long lines: narrower tiles (down to 4 columns) so the staged lines fit
        while (W > 4 && (size_t)(L + 2 * ghost_rows(geo)) * W * sizeof(T) > 200 * 1024) W /= 2;
        int nseg = L / 8;
        const int maxseg = 256 / W > 0 ? 256 / W : 1;
        nseg = nseg > maxseg ? maxseg : (nseg < 1 ? 1 : nseg);
        tu.W = W;
        tu.nseg = nseg;
        const int want = c->opt_impl ? c->opt_impl : 3;
        const int Weff = W < geo.inner ? W : (int)geo.inner;
        tu.impl = (want == 2 && tma_eligible<T>(c, geo, Weff)) ? 2 : (want == 3 && pair_eligible<T>(c, geo, Weff)) ? 3 : 1;
    } else {
        int R = 4096 / L;
        R = R < 32 ? 32 : (R > 128 ? 128 : R);
        while (R > 1 && rows_smem<T>(L, R, ghost_rows(geo)) > 96 * 1024) R /= 2;  // long lines
        int nseg = L / 16;
        const int maxseg = 256 / R > 0 ? 256 / R : 1;
        nseg = nseg > maxseg ? maxseg : (nseg < 1 ? 1 : nseg);
        tu.W = R;
        tu.nseg = nseg;
        const int want = c->opt_impl ? c->opt_impl : 3;
        tu.impl = want == 3 && sizeof(T) == 4 && R % 2 == 0 ? 3 : 1;
    }
    return tu;
}

template <typename T>
int launch_sweep_t(vp_ctx *c, int kick, int dim, double dt, const double *accel, bool tab_ready) {
    const SweepGeo geo = vp_make_geo(c, kick, dim);
    const SweepShift sw{kick, dim, dt, accel, tab_ready, 0};
    SweepTune tu = c->tune[kick][dim];
    if (!tu.valid || (c->opt_impl && tu.impl != c->opt_impl)) tu = default_tune<T>(c, geo);
    if (c->opt_impl == 1) tu.impl = 1;
    if (geo.inner > 1) return launch_cols<T>(c, geo, tu, sw);
    return launch_rows<T>(c, geo, tu, sw);
}

// Autotuner: time candidate tile shapes of one sweep geometry with the
// sweep's own shifts (dt, accel) on a copy of a window at the centre of f --
// whole outer blocks, or where one block exceeds the budget the middle
// columns of every row -- of at most kTuneBytes (larger than L2, so the
// timing sees HBM), and keep the fastest.  The window keeps every line's
// shift class (its offset is a whole number of class periods; a kick window
// reads the shift table from its first spatial point), so the limiter paths
// are timed on the state at hand where the distribution is, not on an empty
// corner of phase space; f is left untouched.  Without room for the copy the
// defaults stay.  Runs once per (kind, axis), never inside a stream capture.
constexpr size_t kTuneBytes = size_t(256) << 20;

template <typename T>
int tune_on(vp_ctx *c, const SweepShift &sw, const SweepGeo &geo, const SweepGeo &sub, SweepTune best);

template <typename T>
int tune_t(vp_ctx *c, int kick, int dim, double dt, const double *accel) {
    const SweepGeo geo = vp_make_geo(c, kick, dim);
    SweepTune best = default_tune<T>(c, geo);
    SweepGeo sub = geo;
    const size_t block = (size_t)geo.L * (size_t)geo.inner * sizeof(T);
    size_t bytes;
    bool pitched = false;
    long long o0 = 0, c0 = 0;  // window offset: outer blocks, columns
    // flattened index of the central cell of spatial axes [a, b)
    auto centre = [&](int a, int b) {
        long long i = 0;
        for (int k = a; k < b; ++k) i = i * c->g.nx[k] + c->g.nx[k] / 2;
        return i;
    };
    auto clampll = [](long long x, long long lo, long long hi) { return x < lo ? lo : (x > hi ? hi : x); };
    // the window's middle: the central spatial cell (and middle velocity)
    const long long o_mid = kick ? centre(0, c->g.dx) * geo.cdiv + geo.cdiv / 2 : centre(0, dim);
    const long long c_mid = kick ? 0 : centre(dim + 1, c->g.dx) * c->NV + c->NV / 2;
    if (block <= kTuneBytes) {
        const long long no = (long long)(kTuneBytes / block);
        sub.outer = no < geo.outer ? no : geo.outer;
        o0 = clampll(o_mid - sub.outer / 2, 0, geo.outer - sub.outer);
        if (!geo.cls_from_inner) o0 -= o0 % geo.cdiv;  // whole spatial points
        bytes = (size_t)sub.outer * block;
    } else {
        long long ni = (long long)(kTuneBytes / ((size_t)geo.L * sizeof(T)));
        if (ni >= 128) ni &= ~127LL;
        if (ni < 1) ni = 1;
        sub.outer = 1;
        sub.inner = ni < geo.inner ? ni : geo.inner;
        o0 = clampll(o_mid, 0, geo.outer - 1);
        if (!geo.cls_from_inner) o0 -= o0 % geo.cdiv;
        // whole velocity periods of the line classes, and 16-byte rows
        const long long per = 4 * (geo.cls_from_inner ? geo.cdiv * geo.cmod : 1);
        c0 = clampll(c_mid - sub.inner / 2, 0, geo.inner - sub.inner);
        c0 -= c0 % per;
        bytes = (size_t)geo.L * (size_t)sub.inner * sizeof(T);
        pitched = true;
    }
    const T *src = static_cast<const T *>(c->f) + (o0 * geo.L * geo.inner + c0);
    void *scratch = nullptr;
    if (cudaMalloc(&scratch, bytes) != cudaSuccess) {
        cudaGetLastError();
        c->tune[kick][dim] = best;
        return VP_OK;
    }
    int rc = VP_OK;
    if (pitched)
        rc = cudaMemcpy2DAsync(scratch, (size_t)sub.inner * sizeof(T), src, (size_t)geo.inner * sizeof(T),
                               (size_t)sub.inner * sizeof(T), (size_t)geo.L, cudaMemcpyDeviceToDevice,
                               c->stream) == cudaSuccess ? VP_OK : vp_fail(c, VP_ECUDA, "tuning copy failed");
    else
        rc = cudaMemcpyAsync(scratch, src, bytes, cudaMemcpyDeviceToDevice, c->stream) == cudaSuccess
                 ? VP_OK : vp_fail(c, VP_ECUDA, "tuning copy failed");
    if (rc == VP_OK) rc = vp_launch_shift_tables(c, kick, 1u << dim, dt, accel);
    if (rc == VP_OK) {
        void *f = c->f;
        c->f = scratch;
        // a kick window starts at spatial point o0 / cdiv
        const long long cls0 = geo.cls_from_inner ? 0 : o0 / geo.cdiv;
        const SweepShift sw{kick, dim, dt, kick ? accel + cls0 : accel, true, cls0};
        rc = tune_on<T>(c, sw, geo, sub, best);
        c->f = f;
    }
    cudaStreamSynchronize(c->stream);
    cudaFree(scratch);
    return rc;
}

// time the candidates of geometry geo on sub (the tuning copy bound as f)
template <typename T>
int tune_on(vp_ctx *c, const SweepShift &sw, const SweepGeo &geo, const SweepGeo &sub, SweepTune best) {
    const int kick = sw.kick, dim = sw.dim;
    int rc = VP_OK;
    constexpr int kMaxCand = 48;
    SweepTune cand[kMaxCand];
    int nc = 0;
    // Small grids (fewer 32-line tiles than two per SM) take narrow tiles of
    // short segments, so that the walk's serial chain is short and every SM has
    // work: 64 x 128 in FP64 had 4 and 8 CTAs (drift 50 us, kick 23 us, the FP64
    // pipe of those SMs busy throughout), 512 x 512 in FP64 16 and 64 (214 and
    // 60 us).  A segment of l cells computes l + 1 interfaces, hence l >= 4.
    const bool small = geo.outer * geo.inner < 64LL * c->sm_count;
    auto add = [&](int impl, int W, int nseg) {
        if (nc < kMaxCand) cand[nc++] = SweepTune{1, impl, W, nseg, 0, 1};
    };
    if (geo.inner > 1) {
        const int impls[3] = {3, 2, 1};
        // lines too long for a 32-column tile take 4-16 columns and more segments
        const bool longl = (size_t)(geo.L + 2 * ghost_rows(geo)) * 32 * sizeof(T) > 200 * 1024;
        for (int ii = 0; ii < 3; ++ii) {
            const int impl = impls[ii], per = impl == 3 ? 2 : 1;
            if (c->opt_impl && impl != c->opt_impl) continue;
            const int w0 = small ? (int)(16 / sizeof(T)) : (longl ? 4 : 32);
            for (int W = w0; W <= (small ? 8 * w0 : (longl ? 16 : 128)); W *= 2)
                for (int nseg = 1; nseg <= (small ? 128 : (longl ? 64 : 8)); nseg *= 2) {
                    const int th = W / per * nseg;
                    if (th > (impl == 3 ? VP_PAIR_THREADS : 512) || nseg > geo.L) continue;
                    if (small) {
                        // segments of 4 to 32 cells, one warp at least where the line has the cells
                        if (nseg * 4 > geo.L || (nseg < 128 && nseg * 64 <= geo.L) || (th < 32 && nseg * 8 <= geo.L))
                            continue;
                    } else if (th < (impl == 3 ? 32 : 64) || (longl && nseg * 8 > geo.L)) {
                        continue;
                    }
                    const int Weff = geo.inner < W ? (int)geo.inner : W;
                    if (impl == 2 && !tma_eligible<T>(c, geo, Weff)) continue;
                    if (impl == 3 && !pair_eligible<T>(c, geo, Weff)) continue;
                    if (impl != 2 && (size_t)(geo.L + 2 * ghost_rows(geo)) * W * sizeof(T) > 200 * 1024)
                        continue;
                    add(impl, W, nseg);
                }
        }
    } else {
        // long lines take fewer lines per CTA (the staged tile must fit) and
        // more segments per line (segments of at least 8 cells; 4 on small grids)
        for (int impl = 1; impl <= 3; impl += 2) {
            const int per = impl == 3 ? 2 : 1;
            if ((c->opt_impl == 1 && impl != 1) || (c->opt_impl == 3 && impl != 3) || (impl == 3 && sizeof(T) != 4))
                continue;
            for (int R = small ? per : 8; R <= (small ? 8 : 128); R *= 2)
                for (int nseg = 1; nseg <= (small ? 256 : 64); nseg *= 2) {
                    const int th = R / per * nseg;
                    if (th > (impl == 3 ? VP_PAIR_THREADS : 512)) continue;
                    if (small) {
                        if (nseg * 4 > geo.L || (nseg < 256 && nseg * 64 <= geo.L) || (th < 32 && nseg * 8 <= geo.L))
                            continue;
                    } else if (th < (impl == 3 ? 32 : 64) || nseg * 8 > geo.L) {
                        continue;
                    }
                    if (rows_smem<T>(geo.L, R, ghost_rows(geo)) > 200 * 1024) continue;
                    add(impl, R, nseg);
                }
        }
    }
    if (nc == 0) {
        c->tune[kick][dim] = best;
        return VP_OK;
    }
    cudaEvent_t e0, e1;
    VP_CUDA_TRY(c, cudaEventCreate(&e0));
    VP_CUDA_TRY(c, cudaEventCreate(&e1));
    float best_ms = 1e30f;
    // Every candidate, then the fastest without the walkers' vote on flat
    // stencils (the same results; the vote pays where f has flat, e.g. empty,
    // regions and costs 7% where it has none: 2D2V Landau drifts 138 -> 128 us).
    // What is timed is today's state, and the limiters' work grows as a run fills
    // its empty space: the TMA pipeline, which walks one line per thread, and the
    // kernels without the vote have to win by 5% and 2%.
    for (int i = 0; i <= nc; ++i) {
        SweepTune t = i < nc ? cand[i] : best;
        if (i == nc) {
            if (t.impl == 2 || !(c->g.mp && c->g.pp)) break;
            t.flat = 0;
        }
        float ms = 1e30f;
        for (int rep = 0; rep < 2; ++rep) {
            cudaEventRecord(e0, c->stream);
            rc = geo.inner > 1 ? launch_cols<T>(c, sub, t, sw) : launch_rows<T>(c, sub, t, sw);
            cudaEventRecord(e1, c->stream);
            if (rc) break;
            const cudaError_t se = cudaEventSynchronize(e1);
            if (se != cudaSuccess) {
                rc = vp_fail(c, VP_ECUDA, "sweep candidate failed: %s", cudaGetErrorString(se));
                break;
            }
            float m = 0.f;
            cudaEventElapsedTime(&m, e0, e1);
            ms = m < ms ? m : ms;
        }
        if (rc) {
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            return rc;
        }
        ms *= t.impl == 2 ? 1.05f : (t.flat ? 1.f : 1.02f);
        if (ms < best_ms) {
            best_ms = ms;
            best = t;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    best.valid = 1;
    c->tune[kick][dim] = best;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

}  // namespace

// The entry points of this unit's precision and order.
void VP_UNIT(vp_sweep_attrs)() { set_attrs<unit_t>(); }

#if VP_SWEEP_ORDER == 7
int VP_UNIT(vp_launch_shift_tables)(vp_ctx *c, int kick, unsigned dims, double dt, const double *accel) {
    const vp_grid &g = c->g;
    TableAxes ax{};
    int most = 0;
    for (int d = 0; d < g.dx; ++d) {
        if (!(dims & (1u << d))) continue;
        const int i = ax.n++;
        const double dvel = (g.vhi[d] - g.vlo[d]) / g.nv[d];
        ax.dim[i] = d;
        ax.nclass[i] = kick ? (int)c->NX : g.nv[d];
        ax.lo[i] = g.vlo[d];
        ax.dvel[i] = dvel;
        ax.h[i] = kick ? dvel : (g.xhi[d] - g.xlo[d]) / g.nx[d];
        // one axis: its own array; several: the components of a field
        ax.accel[i] = kick ? accel + ((dims & (dims - 1)) ? d * c->NX : 0) : nullptr;
        most = ax.nclass[i] > most ? ax.nclass[i] : most;
    }
    const int th = 64;
    const dim3 grid((unsigned)((8LL * most + th - 1) / th), (unsigned)ax.n);
    vp_launch_dep(k_shift_table<unit_t>, grid, th, 0, c->stream, static_cast<LineShift<unit_t> *>(c->d_shift),
                  c->shift_cap, kick, ax, dt, c->wp);
    c->launches++;
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

// whether the sweep along dim reads the context's table (false: its CTAs make
// their own shifts)
bool VP_UNIT(vp_sweep_reads_table)(vp_ctx *c, int kick, int dim) {
    SweepGeo geo = vp_make_geo(c, kick, dim);
    SweepTune tu = c->tune[kick][dim];
    if (!tu.valid || (c->opt_impl && tu.impl != c->opt_impl)) tu = default_tune<unit_t>(c, geo);
    const long long w = geo.inner > 1 ? (geo.inner < tu.W ? geo.inner : tu.W) : (geo.outer < tu.W ? geo.outer : tu.W);
    const long long per = geo.inner > 1 && geo.inner < tu.W ? tu.W / geo.inner : 1;  // blocks per tile
    const long long tiles = geo.inner > 1 ? (geo.outer + per - 1) / per * ((geo.inner + w - 1) / w) : (geo.outer + w - 1) / w;
    return tu.impl == 2 || !own_shifts(c, geo, tiles);
}
#endif

int VP_UNIT(vp_launch_sweep)(vp_ctx *c, int kick, int dim, double dt, const double *accel, bool tab_ready) {
    return launch_sweep_t<unit_t>(c, kick, dim, dt, accel, tab_ready);
}

int VP_UNIT(vp_tune_sweep)(vp_ctx *c, int kick, int dim, double dt, const double *accel) {
    return tune_t<unit_t>(c, kick, dim, dt, accel);
}

#ifdef VP_SWEEP_MAIN
#define VP_DECLARE(U)                                                                                      \
    void vp_sweep_attrs_##U();                                                                             \
    int vp_launch_sweep_##U(vp_ctx *c, int kick, int dim, double dt, const double *accel, bool tab_ready); \
    int vp_tune_sweep_##U(vp_ctx *c, int kick, int dim, double dt, const double *accel)
VP_DECLARE(f32_o5);
VP_DECLARE(f64_o5);
VP_DECLARE(f64_o7);
int vp_launch_shift_tables_f64_o7(vp_ctx *c, int kick, unsigned dims, double dt, const double *accel);
bool vp_sweep_reads_table_f64_o7(vp_ctx *c, int kick, int dim);

int vp_sweep_setup(vp_ctx *c) {
    vp_sweep_attrs_f32_o5();
    vp_sweep_attrs_f32_o7();
    vp_sweep_attrs_f64_o5();
    vp_sweep_attrs_f64_o7();
    VP_CUDA_TRY(c, cudaGetLastError());
    return VP_OK;
}

int vp_launch_shift_tables(vp_ctx *c, int kick, unsigned dims, double dt, const double *accel) {
    return c->g.precision == VP_F32 ? vp_launch_shift_tables_f32_o7(c, kick, dims, dt, accel)
                                    : vp_launch_shift_tables_f64_o7(c, kick, dims, dt, accel);
}

int vp_launch_shift_tables_f32(vp_ctx *c, int kick, unsigned dims, double dt, const double *accel) {
    return vp_launch_shift_tables_f32_o7(c, kick, dims, dt, accel);
}

bool vp_sweep_reads_table(vp_ctx *c, int kick, int dim) {
    return c->g.precision == VP_F32 ? vp_sweep_reads_table_f32_o7(c, kick, dim)
                                    : vp_sweep_reads_table_f64_o7(c, kick, dim);
}

int vp_launch_sweep(vp_ctx *c, int kick, int dim, double dt, const double *accel, bool tab_ready) {
    if (c->g.precision == VP_F32)
        return c->g.order == 7 ? vp_launch_sweep_f32_o7(c, kick, dim, dt, accel, tab_ready)
                               : vp_launch_sweep_f32_o5(c, kick, dim, dt, accel, tab_ready);
    return c->g.order == 7 ? vp_launch_sweep_f64_o7(c, kick, dim, dt, accel, tab_ready)
                           : vp_launch_sweep_f64_o5(c, kick, dim, dt, accel, tab_ready);
}

int vp_tune_sweep(vp_ctx *c, int kick, int dim, double dt, const double *accel) {
    if (c->tune[kick][dim].valid) return VP_OK;
    if (c->g.precision == VP_F32)
        return c->g.order == 7 ? vp_tune_sweep_f32_o7(c, kick, dim, dt, accel)
                               : vp_tune_sweep_f32_o5(c, kick, dim, dt, accel);
    return c->g.order == 7 ? vp_tune_sweep_f64_o7(c, kick, dim, dt, accel)
                           : vp_tune_sweep_f64_o5(c, kick, dim, dt, accel);
}
#endif

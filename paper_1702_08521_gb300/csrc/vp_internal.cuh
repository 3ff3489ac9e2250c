// vp_internal.cuh -- shared declarations of the CUDA library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdarg>
#include <cstdio>

#include "vlasov.h"

// Per line class (one velocity index for a drift, one spatial cell for a
// kick): the integer shift n, the direction sigma = sign(zeta), the CFL number
// nu = |zeta| and the CSL weights w_k(nu) on the upwind-ordered stencil
// u[-3..3] (u[0] = upwind cell of the interface).  For CSL5 w[0] = w[6] = 0.
template <typename T>
struct __align__(16) LineShift {
    T w[7];
    T nu;
    int n;
    int sigma;
};

// Geometry of one sweep: f viewed as [outer][L][inner].
// Division of 32-bit unsigned values by a divisor (not 0) fixed before the launch
// (Granlund & Montgomery 1994, Fig. 4.1): with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, n / d = (t + ((n - t) >> s1)) >> s2
// where t = high word of m n, s1 = min(l, 1), s2 = max(l - 1, 0).
struct FastDiv {
    unsigned d, m;
    int s1, s2;
};

inline FastDiv make_fastdiv(unsigned d) {
    int l = 0;
    while (l < 32 && (1ull << l) < d) ++l;
    FastDiv f;
    f.d = d;
    f.m = (unsigned)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
    f.s1 = l < 1 ? l : 1;
    f.s2 = l > 1 ? l - 1 : 0;
    return f;
}

#ifdef __CUDACC__
__host__ __device__ __forceinline__ unsigned fdiv(unsigned n, const FastDiv &f) {
#ifdef __CUDA_ARCH__
    const unsigned t = __umulhi(n, f.m);
#else
    const unsigned t = (unsigned)(((unsigned long long)n * f.m) >> 32);
#endif
    return (t + ((n - t) >> f.s1)) >> f.s2;
}
__host__ __device__ __forceinline__ unsigned fmod_u(unsigned n, const FastDiv &f) { return n - fdiv(n, f) * f.d; }

// The lines along one axis of f viewed as [outer][L][inner], `lines` = outer inner
// of them, and their classes: of the inner index (from_inner) or the outer one,
// divided by cdiv, modulo cmod.  Multiplications in place of divisions for fewer
// than 2^32 lines (the indices and cdiv are then below 2^32 too), 64-bit ones beyond.
struct LineShape {
    long long lines, inner, cdiv;
    int L, periodic, from_inner;
    unsigned cmod;
    FastDiv fd_inner, fd_cdiv, fd_cmod;

    void prepare() {
        const bool narrow = lines < (1LL << 32);
        fd_inner = make_fastdiv(narrow ? (unsigned)inner : 1u);
        fd_cdiv = make_fastdiv(narrow ? (unsigned)cdiv : 1u);
        fd_cmod = make_fastdiv(cmod);
    }
    // the line's class; base: element of its first cell
    __host__ __device__ __forceinline__ unsigned place(long long line, long long &base) const {
        if (lines < (1LL << 32)) {
            const unsigned o = fdiv((unsigned)line, fd_inner), c = (unsigned)line - o * (unsigned)inner;
            base = (long long)o * L * inner + c;
            return from_inner ? fmod_u(fdiv(c, fd_cdiv), fd_cmod) : fdiv(o, fd_cdiv);
        }
        const long long o = line / inner, c = line - o * inner;
        base = o * L * inner + c;
        return (unsigned)(from_inner ? c / cdiv % cmod : o / cdiv);
    }
};
#endif

// Programmatic dependent launch: a kernel launched by vp_launch_dep may start
// while the kernel before it on the stream is still finishing.  It calls
// dep_wait() before its first access to memory that another launch wrote or still
// reads (the grids before it are then complete and visible) and dep_launch() to
// let the next one start.  Its pointers carry no __restrict__, which would let
// the compiler move their loads above the wait.  A step on a small grid is a chain of kernels of
// 2-20 us, each of which waited ~1 us for the launch of the next: 1D1V Landau
// 64 x 128 FP64 36.4 -> 33.8 us a step, two-stream 256 x 1024 499 -> 454,
// 512 x 512 FP64 sweeps 78.5 -> 73.2.  Only grids of at most one CTA per SM let
// the next one in early; from larger ones it would take the slots of CTAs that
// still have work (two-stream 564, a learned 2D2V step 346 -> 361), so there the
// launch alone overlaps.
#ifdef __CUDACC__
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_launch() {
    unsigned sms;
    asm("mov.u32 %0, %%nsmid;" : "=r"(sms));
    if (gridDim.x * gridDim.y <= sms) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KA, typename... A>
inline void vp_launch_dep(void (*kernel)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = st != nullptr && st != cudaStreamLegacy ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, KA(args)...);
}
#endif

struct SweepGeo {
    long long outer, inner;
    int L;
    int periodic;
    // class of a line: cls_from_inner ? (c / cdiv) % cmod : o / cdiv
    int cls_from_inner;
    long long cdiv, cmod;
    // column-kernel tile (W columns x full line), row-kernel lines per CTA
    int W, nseg, R;
    int kblk;  // column kernel: whole outer blocks per tile (W = kblk inner), or 1
    int vec;   // column kernel: elements per staged piece
    // divisors of the launch: cdiv, cmod, tiles per outer index, W (or R),
    // nseg, L, 16-byte pieces per tile row
    FastDiv fd_cdiv, fd_cmod, fd_tpo, fd_w, fd_nseg, fd_l, fd_wv, fd_w2, fd_inner;
    unsigned tpo;
};

// zero rows staged on each side of an outflow line (a shift |n| <= VP_GHOST - 4
// walks the line without bounds handling)
#define VP_GHOST 8

// tile configuration of one sweep geometry (chosen by the autotuner)
struct SweepTune {
    int valid;
    int impl;   // 1: staged loads (k_sweep_cols / k_sweep_rows), 2: TMA pipeline,
                // 3: staged loads with two lines per thread (FP32 strided sweeps)
    int W, nseg, ctas_per_sm;
    int flat;   // the walkers vote on flat stencils (1) or leave the vote out (0)
};

// tile of the unsplit step (T1 x1 rows x T2 x2 cells x TV velocity cells,
// `threads` per CTA), one per halo width (4 or 8 cells)
struct UnsplitTune {
    int valid;
    int T1, T2, TV, threads;
};

struct LimParams {
    double alpha;
    int mp, pp;
};

// CSL weight polynomials: w_k(nu) = sum_j c[j][k] nu^j.
struct WPoly {
    double c[7][7];
    int nterm;  // 5 or 7 polynomial terms
};

struct vp_graph_cache {
    cudaGraphExec_t exec;
    double dt;
    int split;
    void *f;
    double *acc;
    long long per_step;  // kernels in one captured step
    const float *wts;    // network of the learned drifts (NULL: plain step)
    int valid;
};

struct vp_ctx {
    vp_grid g;
    cudaStream_t stream;
    int device, sm_count;
    long long NX, NV, ncell;
    int esize;
    void *f;
    WPoly wp;
    // library-owned device buffers (the small ones in one allocation, d_arena)
    void *d_arena;
    void *d_shift;
    long long shift_cap;
    double *d_rho, *d_phi, *d_acc;      // diagnostics scratch
    double *d_rho_s;                    // step scratch
    double2 *d_fft;
    double *d_green;                    // periodic: S / lambda(k)
    double2 *d_ghat;                    // isolated: DFT of the padded Green function
    double2 *d_roots, *roots[3];        // roots of unity of the transformed axes (roots[d]: axis d's n)
    double *d_conv;                     // periodic 1D: convolution kernels of phi and the acceleration
    long long MT;
    int m[3];
    double *d_part;                     // diagnostics partial sums [NX * 6]
    double *d_diag;                     // VP_NDIAG doubles
    void *d_vw;                         // kinetic-energy weights: velocity rows, then the last axis
    double vw_unit;                     // the power of two they are divided by
    double *d_diagblk;                  // diagnostics: per-block results (d_diagctr: finished blocks)
    unsigned *d_diagctr;
    int *d_flag;                        // non-finite flag
    long long launches;
    int *d_status;                      // device-side error word (bounded waits)
    void *d_netfrag;                    // network weights in MMA fragment order (allocated on first use)
    void *d_learn_out;                  // learned sweep: the updated lines (allocated on first use)
    int learned_ready;                  // learned-sweep buffers allocated, kernel attributes set
    int opt_impl;                       // 0 auto, 1 staged, 2 TMA
    int opt_autotune;                   // 1: time candidate tiles on first use
    unsigned opt_wait_limit;            // iterations of each bounded device-side wait
    SweepTune tune[2][3];               // [kick][dim]
    UnsplitTune utune[2];               // unsplit step, [halo of 8 cells]
    vp_graph_cache graph;
    char err[256];
};

// error helpers
int vp_fail(vp_ctx *c, int code, const char *fmt, ...);

// line geometry of the sweep (kick, dim): lines of L cells at stride
// `inner`, `outer` blocks of them, and the class of a line (its velocity index
// for drifts, its spatial point for kicks) that selects its shift
inline SweepGeo vp_make_geo(const vp_ctx *c, int kick, int dim) {

    const vp_grid &g = c->g;
    SweepGeo geo{};
    if (!kick) {
        long long outer = 1, inner = c->NV, vstride = 1;
        for (int k = 0; k < dim; ++k) outer *= g.nx[k];
        for (int k = dim + 1; k < g.dx; ++k) inner *= g.nx[k];
        for (int k = dim + 1; k < g.dv; ++k) vstride *= g.nv[k];
        geo.outer = outer;
        geo.inner = inner;
        geo.L = g.nx[dim];
        geo.periodic = g.xbc == VP_BC_PERIODIC;
        geo.cls_from_inner = 1;
        geo.cdiv = vstride;
        geo.cmod = g.nv[dim];
    } else {
        long long vouter = 1, inner = 1;
        for (int k = 0; k < dim; ++k) vouter *= g.nv[k];
        for (int k = dim + 1; k < g.dv; ++k) inner *= g.nv[k];
        geo.outer = c->NX * vouter;
        geo.inner = inner;
        geo.L = g.nv[dim];
        geo.periodic = 0;
        geo.cls_from_inner = 0;
        geo.cdiv = vouter;
        geo.cmod = 1;
    }
    geo.fd_cdiv = make_fastdiv((unsigned)geo.cdiv);
    geo.fd_cmod = make_fastdiv((unsigned)geo.cmod);
    return geo;
}

#define VP_CUDA_TRY(ctx, call)                                                         \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            return vp_fail((ctx), VP_ECUDA, "%s: %s", #call, cudaGetErrorString(e_));  \
    } while (0)

// launchers implemented in the kernel files; all enqueue on ctx->stream
// the shift tables of the sweeps along the axes of the bit set `dims`, at d_shift
// + dim * shift_cap; accel: of one axis its array, of several the whole field
int vp_launch_shift_tables(vp_ctx *c, int kick, unsigned dims, double dt, const double *accel);
// the same in FP32 whatever the grid's precision (the learned part's kernels)
int vp_launch_shift_tables_f32(vp_ctx *c, int kick, unsigned dims, double dt, const double *accel);
bool vp_sweep_reads_table(vp_ctx *c, int kick, int dim);
// the context stream is being captured into a graph (no synchronising calls)
bool vp_capturing(const vp_ctx *c);
// buffers and kernel attributes of the learned sweep (outside any stream capture)
int vp_learned_prepare(vp_ctx *c);
// one learned drift along dim from fin to fout (distinct arrays of f's size);
// net: make the network operands from wts first; tab_ready: the drift's shift table is made already
int vp_learned_drift_io(vp_ctx *c, int dim, double dt, const float *wts, int use_net, const float *fin,
                        float *fout, bool net, bool tab_ready);
// RK-MPP5 sweeps: kernel attributes once per process, one sweep (table + fused stages)
int vp_rk_setup();
int vp_launch_rk_sweep(vp_ctx *c, int kick, int dim, double dt, const double *accel);
// one SL sweep; tab_ready: its shift table is made already, else it makes it
// where it needs one
int vp_launch_sweep(vp_ctx *c, int kick, int dim, double dt, const double *accel, bool tab_ready);
// autotune sweep (kick, dim) at its own shifts (dt, accel); outside stream capture only
int vp_tune_sweep(vp_ctx *c, int kick, int dim, double dt, const double *accel);
int vp_launch_moment(vp_ctx *c, double *rho);
// phi may be NULL
int vp_launch_poisson(vp_ctx *c, const double *rho, double *phi, double *acc);
int vp_launch_diag(vp_ctx *c, int mode, double *out_dev);
int vp_launch_init(vp_ctx *c, int kind, const double *p, int np);
// bytes of the field solve's and the diagnostics' tables in the arena
struct FieldSizes {
    size_t green, roots, conv, weights, diagblk;
};
FieldSizes vp_field_sizes(const vp_ctx *c);
int vp_field_setup(vp_ctx *c);          // fills those tables, the isolated Green function (at create)
// CSL weight polynomials of the given order (5 or 7), from the definition of the SL flux
WPoly vp_csl_weight_polys(int order);
// learned flux correction network: 25 features, 3 hidden layers of 32
#define VP_NET_FEATURES 25
#define VP_NET_HIDDEN 32
// analytic initial condition into any f array of grid g (precision from g)
int vp_launch_init_ptr(void *f, const vp_grid &g, int kind, const double *p, int np, cudaStream_t st);
int vp_sweep_setup(vp_ctx *c);          // kernel attributes (at create)

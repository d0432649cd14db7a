// Fused stream-collide kernel (one launch per time step over every stored
// cell of every instance) and its launcher with the autotuner's variants.
#include "lbm_collide.cuh"

namespace lbm {

constexpr int LINE_CELLS = 64;  // a cache line of 16-bit populations, two of FP32

// Where the populations exceed the L2, one block of every AHEAD_CELLS cells has
// the populations of as many cells fetched into the L2, AHEAD_DIST cells before
// the blocks reach them: the loads of a block wait for the L2 instead of the
// memory, and the bytes in flight are not bound by the warps' registers (without,
// FP16 issued 0.55 and stalled on loads for half of its time at 43 warps an SM).
// One bulk prefetch per direction and block of 128 cells is too many requests for
// FP16 (364 -> 402 us per step of 96 uneven tubes, FP32 481 -> 468); of 512, 2,048,
// 4,096, 8,192 cells: FP16 358, 351, 360, 366, FP32 467, 462, 462, 473.  8,192 to
// 32,768 cells ahead are alike, 131,072 slower (517 with single blocks): what is
// fetched so early takes the place of what neighbouring planes still need.  Before
// and after: 96 uneven tubes 481 -> 462 (FP16 364 -> 348), aorta 215.5 -> 212.4 (FP16
// 187.6 -> 184.0).  The mask comes from the host: a division per thread costs FP16,
// which is bound by instruction issue then, all of the gain.
constexpr int AHEAD_CELLS = 2048, AHEAD_DIST = 16384;
// The blocks that fetch, as a mask of the block index (0: none).
int ahead_mask(const KParams &p, int block, int cpt) {
    if (!p.keep || cpt != 1 || p.n % LINE_CELLS) return 0;
    int per = 1;
    while (2 * per * block <= AHEAD_CELLS) per *= 2;
    return per - 1;
}

// One base pointer per direction of the input and output population arrays
// (f_i = f + i N, structure of arrays), passed in the kernel's parameter
// space: every pull and store then forms its address with one wide
// multiply-add from a constant-bank operand.
template <class S> struct PopDirs {
    const S *in[NQ];
    S *out[NQ];
    __device__ __forceinline__ S *operator()(int i, int c) const { return out[i] + c; }
};

// ---------------------------------------------------------------------------
// Fused stream-collide.  For each fluid cell x and direction i the pulled
// population is f*_i(x - e_i) (or f*_opp(i)(x) when x - e_i is a rigid wall:
// halfway bounce-back).  Then P = c_s^2 sum f, j = sum e f, v = j + b/2
// (Eqs. rho, v), f^eq (Eq. feq), the forcing F_i (Eq. f) and BGK relaxation
// (Eq. fi).  With s = f - w: sum f = 1 + sum s, j = sum e s, and
// f^eq_i - w_i = w_i (K + 3 e.v + 9/2 (e.v)^2), K = sum s - 3/2 v^2.
//
// Arithmetic per cell, arranged for few instructions (the 16-bit storage
// variants are bound by instruction issue, not by bytes):
// * pull: the pull source of direction i lies on one of 8 neighbouring
//   lattice lines (or the own row), at x - e_ix; a bounce-back link instead
//   reads the opposite population of the own cell, which in this layout is
//   f_i + (opp(i) - i) N + c with opp(i) - i = +-1, so one select of a
//   32-bit index per direction covers both cases;
// * moments from the sums and differences of the 9 opposite pairs;
// * relaxation per opposite pair (i, i'): with A = omega w (K + 9/2 (e.v)^2)
//   and B = 3 omega w e.v, s*_i = (1 - omega) s_i + A + B and
//   s*_i' = (1 - omega) s_i' + A - B; Guo's F_i splits the same way into the
//   pair-symmetric part w (1 - omega/2) (9 (e.v)(e.b) - 3 v.b) and the
//   antisymmetric 3 w (1 - omega/2) e.b.  The forcing is evaluated only by
//   warps that hold a band cell (a warp-uniform branch).
//
// Occupancy request to ptxas (template parameter MINB: at least MINB resident
// 256-thread blocks per SM).  CPT > 1 gives each thread CPT independent
// cells, one grid stride apart, whose loads are all issued before any of
// them is consumed.  The variants are kept for the run-time autotuner.
// desc = 1 maps the blocks to the cells in descending order, so that a
// launch starts on the lines the previous kernel touched last (still in L2).
// The launch covers the stored cells [c0, c1), its blocks beginning on whole
// cache lines (a batch in two parts, the second from an odd cell: 500 us per
// step, from its cache line 486); the launch with bump = 1 advances the step
// counter.
// EARLY: launched while its predecessor, the boundary kernel, still runs (see
// launch_stream_collide); only tables that no step writes are read before the
// wait.
// LARGE: the populations exceed the L2 (the rule stands in lbm_create); they are
// fetched ahead and their stores stay in the L2.  A kernel of its own: with both switched at run time
// lattices that fit took 1 to 2.5 % longer (tubes of 508,000, 643,000, 1.03 M cells
// FP32 21.2 -> 21.5, 26.3 -> 26.8, 37.1 -> 37.6 us per step, FP16 18.9 -> 19.2, 20.6 -> 21.1,
// 27.8 -> 28.6), about half from either.
template <class S, int MINB, int CPT, bool EARLY, bool LARGE>
__global__ void __launch_bounds__(256, MINB)
    k_stream_collide(const __grid_constant__ PopDirs<S> d, const __grid_constant__ KParams p, int desc, int c0,
                     int c1, int bump, int ahead) {
    using R = typename Storage<S>::R;
    const int bid = desc ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int t = (c0 & ~(LINE_CELLS - 1)) + bid * blockDim.x + threadIdx.x;
    const int stride = gridDim.x * blockDim.x;
    if (!EARLY && bump && t == c0 && p.step) *p.step += 1;  // the step index t_n seen by the boundary kernels
    const int N = (int)p.n;  // 19 N < 2^31 is checked at creation
    if (LARGE && CPT == 1 && threadIdx.x < NQ && ahead && (bid & ahead) == 0) {
        const int s = t - (int)threadIdx.x + (desc ? -AHEAD_DIST : AHEAD_DIST), n = (ahead + 1) * (int)blockDim.x;
        if (s >= c0 && s < c1 && s + n <= N)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(d.in[0] + ((long long)threadIdx.x * N + s)),
                         "r"((unsigned)(n * sizeof(S))));
    }
    R f[CPT][NQ];
    R om[CPT];
    uint32_t fl[CPT];
#pragma unroll
    for (int u = 0; u < CPT; u++) {
        const int c = t + u * stride;
        fl[u] = c >= c0 && c < c1 ? __ldg(&p.flags[c]) : 0u;
        om[u] = R(0);
        const bool active = (fl[u] & FL_ACTIVE) != 0;
        if (!EARLY && !active) continue;
        int4 h0 = {}, h1 = {}, h2 = {}, h3 = {};
        if (!EARLY || active) {
            const int4 *row = reinterpret_cast<const int4 *>(p.rows + find_row(p, c));
            h0 = __ldg(row);
            h1 = __ldg(row + 1);
            h2 = __ldg(row + 2);
            h3 = __ldg(row + 3);
        }
        if (EARLY) {
            wait_for_previous();
            let_next_start();
            if (bump && t == c0 && p.step) *p.step += 1;
            if (!active) continue;
        }
        // h0 = {off, x0, len, inst}, h1 = {y, z, nb0, nb1}, h2 = {nb2..nb5}, h3 = {nb6, nb7, nb8, pad}
        om[u] = omega_of<R>(p, h0.w);
        const int x = h0.y + (c - h0.x);
        const int line[9] = {h1.z + x, h1.w + x, h2.x + x, h2.y + x, c, h2.w + x, h3.x + x, h3.y + x, h3.z + x};
        f[u][0] = Storage<S>::ld(d.in[0] + c);
#pragma unroll
        for (int i = 1; i < NQ; i++) {
            const int src = line[nbk(i)] - cx(i);               // pull from x - e_i
            const int own = c + ((i & 1) ? N : -N);              // f_opp(i)(x) = f_i + (opp(i) - i) N + x
            const int idx = ((fl[u] >> i) & 1u) ? own : src;     // halfway bounce-back
            f[u][i] = Storage<S>::ld(d.in[i] + idx);
        }
    }
#pragma unroll
    for (int u = 0; u < CPT; u++) {
        const int c = t + u * stride;
        const bool band = (fl[u] & (FL_ACTIVE | FL_BAND)) == (FL_ACTIVE | FL_BAND);
        if (__any_sync(0xffffffffu, band)) {
            if (fl[u] & FL_ACTIVE) collide_store<S, R, true, LARGE>(d, p, f[u], om[u], fl[u], c);
        } else {
            if (fl[u] & FL_ACTIVE) collide_store<S, R, false, LARGE>(d, p, f[u], om[u], fl[u], c);
        }
    }
}

// ---------------------------------------------------------------------------
// launcher

// variants: {min blocks per SM, cells per thread}
static const int kVariants[SC_VARIANTS][2] = {{6, 1}, {8, 1}, {5, 1}, {4, 2}, {3, 2}};

int stream_collide_min_blocks(int variant) { return kVariants[variant][0]; }
int stream_collide_cells_per_thread(int variant) { return kVariants[variant][1]; }

template <class S> static PopDirs<S> pop_dirs(const void *fin, void *fout, long long n) {
    PopDirs<S> d;
    for (int i = 0; i < NQ; i++) {
        d.in[i] = static_cast<const S *>(fin) + (size_t)i * (size_t)n;
        d.out[i] = static_cast<S *>(fout) + (size_t)i * (size_t)n;
    }
    return d;
}

template <class S, int MINB, int CPT>
static void launch(int grid, int block, cudaStream_t s, const void *fin, void *fout, const KParams &p, int desc, int c0,
                   int c1, int bump, int ahead) {
    const auto k = p.keep ? k_stream_collide<S, MINB, CPT, false, true> : k_stream_collide<S, MINB, CPT, false, false>;
    k<<<grid, block, 0, s>>>(pop_dirs<S>(fin, fout, p.n), p, desc, c0, c1, bump, ahead);
}

template <class S>
static cudaError_t early_launch(int grid, int block, cudaStream_t s, const void *fin, void *fout, const KParams &p, int desc,
                                int c0, int c1, int bump, int ahead) {
    const auto k = p.keep ? k_stream_collide<S, 6, 1, true, true> : k_stream_collide<S, 6, 1, true, false>;
    return launch_early(k, dim3(grid), dim3(block), s, pop_dirs<S>(fin, fout, p.n), p, desc, c0, c1, bump, ahead);
}

cudaError_t launch_stream_collide(int prec, const void *fin, void *fout, const KParams &p, int block,
                                  int variant, cudaStream_t s, int desc, int c0, int c1, int bump, bool early) {
    if (c1 < 0) c1 = p.cells;
    if (c1 <= c0) return cudaSuccess;
    if (block % 32) return cudaErrorInvalidValue;  // whole warps: the forcing branch is a warp vote
    const int cpt = kVariants[variant][1];
    const int grid = (int)((c1 - (c0 & ~(LINE_CELLS - 1)) + (long long)block * cpt - 1) / ((long long)block * cpt));
    const int ahead = ahead_mask(p, block, cpt);
    if (early && variant == 0 && prec != 3) {  // FP64 has no one-launch boundary kernel
        cudaError_t e = cudaSuccess;
        DISPATCH_F32(prec, (e = early_launch<S>(grid, block, s, fin, fout, p, desc, c0, c1, bump, ahead)));
        return e;
    }
    switch (variant) {
    case 1: DISPATCH(prec, (launch<S, 8, 1>(grid, block, s, fin, fout, p, desc, c0, c1, bump, ahead))); break;
    case 2: DISPATCH(prec, (launch<S, 5, 1>(grid, block, s, fin, fout, p, desc, c0, c1, bump, ahead))); break;
    case 3: DISPATCH(prec, (launch<S, 4, 2>(grid, block, s, fin, fout, p, desc, c0, c1, bump, ahead))); break;
    case 4: DISPATCH(prec, (launch<S, 3, 2>(grid, block, s, fin, fout, p, desc, c0, c1, bump, ahead))); break;
    default: DISPATCH(prec, (launch<S, 6, 1>(grid, block, s, fin, fout, p, desc, c0, c1, bump, ahead))); break;
    }
    return cudaGetLastError();
}

}  // namespace lbm

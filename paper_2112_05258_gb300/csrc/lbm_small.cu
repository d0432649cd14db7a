// Many steps of small lattices in one launch (no wall nodes).  A thread-block
// cluster takes one instance and advances it n steps, its populations staying
// in L2; the hardware cluster barrier separates the steps, so a step costs
// neither launches nor the gaps between them.  Lattices that are too large for
// clusters of 16 blocks, up to what the shared memory of all SMs takes (about
// 390,000 cells), are one cooperative grid with a barrier in global memory.
//
// Work of the C blocks of an instance (grid: of all instances) with B 0D boundaries:
//   * block k < B owns boundary k: it collides the cells of its first fluid
//     layer, sums flow and pressure over them (from registers), takes the 0D
//     step and writes the ghosts of t_{n+1}.  Ghosts are pulled only by
//     first-layer cells, i.e. by the same block in the next step, and the
//     moments never leave it;
//   * the blocks k >= B share the other cells.
// Both only need the other blocks' populations of the step before, so there is
// one cluster barrier per step, and the 0D work runs beside the bulk.
// The pull sources of every cell (18 offsets into the population buffer, the
// bounce-back and the row lookup resolved) are laid out once per launch in
// shared memory: the loop starts its loads without any other lookup.
//
// Same device functions and the same summation order as the one-step kernels
// (collide_store, the 256-wide trees and partial sums, bc_step, ghost_change):
// the trajectory is the same bit for bit.
//
// Bound by latency: the boundary block's chain decides.  An FP64 operation takes
// 64 cycles on this part, a division about 700.  For the 24x24x64 tube (12,896
// cells, FP32) about 1,500 cycles for the pulls, 1,600 collision and the layer's
// terms, 1,400 trees, 2,300 means and 0D step, 1,300 ghosts.  Kept out of the
// chain: the cluster barrier (arrival, which waits for a warp's stores, as soon
// as a warp is not needed for the sums; the ghosts are written after it), all
// that does not depend on the step's flow (inlet velocities, elastance terms,
// state and waveform stores: on threads of their own), divisions by the layer's
// area and the compliance (quotient).
// A step: 12.4 -> 4.1 us for that tube, 12.1 -> 3.5 us for 2,400 cells (FP32), 20.7
// -> 10.1 us in FP64 (whose collision is bound by the FP64 pipe).
//
// The grid: its barrier makes a step 0.4 us longer than a cluster's (3.9 against
// 3.5 us for 14,112 cells).  Its latency is kept out of the boundary block's
// chain: one thread outside the 0D step announces the layer's populations as soon
// as they are stored, and polls beside the ghosts (a fence in each thread and a
// poll after the ghosts: 5.1 us).  Bulk blocks take about 2.05 us and 2.6 ns a
// cell (L2 and issue).
// A step of one-step kernels -> of the grid, FP32: 49,928 cells 9.4 -> 5.6 us,
// 106,920 11.6 -> 6.8, 176,407 12.4 -> 7.2, 323,176 14.5 -> 10.8; 16 instances of
// 14,112 10.4 (clusters) -> 6.9; FP64: 12,896 21.7 -> 18.1, 176,407 64.8 -> 47.4.
#include <cooperative_groups.h>

#include <algorithm>

#include "lbm_collide.cuh"
#include "lbm_ghost.cuh"

namespace lbm {

namespace {

// Populations are read with plain loads: they are written during the launch,
// so not through the read-only path.
template <class S> struct PlainLoad;
template <> struct PlainLoad<float> {
    static __device__ __forceinline__ float ld(const float *p) { return *p; }
};
template <> struct PlainLoad<double> {
    static __device__ __forceinline__ double ld(const double *p) { return *p; }
};
template <> struct PlainLoad<__half> {
    static __device__ __forceinline__ float ld(const __half *p) { return __half2float(*p); }
};
template <> struct PlainLoad<__nv_bfloat16> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
};

template <class S> struct OneBase {
    S *f;
    int N;
    __device__ __forceinline__ S *operator()(int i, int c) const { return f + (i * N + c); }  // 19 N < 2^31
};

// offset in the population buffer that direction i of cell c is pulled from
__device__ __forceinline__ void pull_offsets(const KParams &p, int c, uint32_t fl, int *tab, int stride) {
    const int N = (int)p.n;
    const int r = find_row(p, c);
    const RowInfo &ri = p.rows[r];
    const int x = ri.x0 + (c - ri.off);
#pragma unroll
    for (int i = 1; i < NQ; i++) {
        const int src = (nbk(i) == 4 ? c : ri.nb[nbk(i)] + x) - cx(i);
        tab[(i - 1) * stride] = ((fl >> i) & 1u) ? opp(i) * N + c : i * N + src;
    }
}

template <class R> struct FirstLayer {  // of one first-layer cell: velocity and (sum s) / 3; v_0 of its closure (LV)
    R v[3], p;
};

constexpr int PULLS = NQ - 1;

// The barrier between the steps, arrived at by every warp and waited for later:
// the hardware barrier of a cluster, or, for a whole grid (cooperative launch:
// all blocks are resident), a counter in global memory.  There one thread
// outside the 0D step adds the block, after a __syncthreads() behind its stores,
// polls the counter and releases the block's warps through an mbarrier.  Every
// wait is bounded: when one runs out (seconds; a step takes microseconds) the
// status word says so and the block leaves its loop.
template <bool GRID, int THREADS> struct StepBarrier;
template <int THREADS> struct StepBarrier<false, THREADS> {
    struct Shared {};
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    __device__ StepBarrier(Shared &, const SmallKParams &, unsigned *) {}
    __device__ __forceinline__ void arrive() { cluster.barrier_arrive(); }
    __device__ __forceinline__ bool wait() {
        cluster.barrier_wait();
        return true;
    }
};
template <int THREADS> struct StepBarrier<true, THREADS> {
    struct Shared {
        unsigned long long bar;
        int failed;
    };
    static constexpr int POLLER = THREADS - 32;
    static constexpr int TRIES = 1 << 30;  // a warp never gives up before the polling thread has
    Shared &s;
    const int polls;
    unsigned *count, *status, target = 0, phase = 0;
    __device__ StepBarrier(Shared &sh, const SmallKParams &sp, unsigned *st)
        : s(sh), polls(sp.polls), count(sp.meet), status(st) {
        if (threadIdx.x == 0) {
            s.failed = 0;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(address()) : "memory");
        }
    }
    __device__ __forceinline__ uint32_t address() const { return (uint32_t)__cvta_generic_to_shared(&s.bar); }
    // after a __syncthreads() behind the block's stores
    __device__ __forceinline__ void arrive() {
        if (threadIdx.x == POLLER) {
            __threadfence();
            atomicAdd(count, 1u);
        }
    }
    __device__ __forceinline__ bool wait() {
        target += gridDim.x;
        if (threadIdx.x == POLLER) {
            unsigned v = 0;
            int k = 0;
            do asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            while ((int)(v - target) < 0 && ++k < polls);
            if (k == polls) {
                atomicOr(status, 4u);
                s.failed = 1;
            }
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(address()) : "memory");
        }
        uint32_t done = 0;
        for (int k = 0; k < TRIES && !done; k++)
            asm volatile(
                "{\n.reg .pred p;\n"
                "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                "selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(address()), "r"(phase)
                : "memory");
        phase ^= 1u;
        return done && !*(volatile int *)&s.failed;
    }
};

}  // namespace

// Shared memory of a block.  Boundary block: per first-layer cell the pull
// table, the cell, its moments and its closure velocity; per link its
// destination offset and {direction, first-layer index, node}; per boundary
// node its profile and the prescribed velocity.  Bulk block: pull table and cell per cell.
size_t small_smem_boundary(int n_xf, int n_links, int n_nodes, bool f64) {
    const size_t r = f64 ? 8 : 4;
    return (size_t)n_xf * (PULLS * 4 + 4 + 8 * r) + (size_t)n_links * 8 + (size_t)n_nodes * (24 + 2 * r) + 64;
}
size_t small_smem_bulk(int cells) { return (size_t)cells * (PULLS * 4 + 4) + 64; }
size_t small_smem_grid(int cells, bool f64) { return (size_t)cells * (PULLS * 4 + 4 + (f64 ? 8 : 4)) + 64; }

// GRID: one grid over all instances instead of a cluster per instance (larger
// lattices): block b < n_bc_total owns boundary b, the others share the bulk.
template <class S, int THREADS, bool GRID>
__global__ void __launch_bounds__(THREADS, 1) k_small_steps(S *f0, S *f1, KParams p, BcKParams q, SmallKParams sp) {
    using R = typename Storage<S>::R;
    __shared__ typename StepBarrier<GRID, THREADS>::Shared s_bar;
    StepBarrier<GRID, THREADS> barrier(s_bar, sp, p.status);
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ double sQ[THREADS], sP[THREADS], s_part[2 * SMALL_MAX_RED], s_cos, s_sin;
    __shared__ BcStepResult s_r;
    __shared__ BcParam s_P;
    __shared__ BcState s_st;
    __shared__ Ahead s_a;
    __shared__ double s_area, s_inv_area, s_third;  // n_xf, 1 / n_xf and n_xf / 3
    __shared__ int s_euler;
    __shared__ R s_dir[NQ][4];  // e_i and w_i
    // C blocks share the instances inst .. of which the first nb own boundaries b0 ..
    const int C = GRID ? (int)gridDim.x : sp.cluster, rank = (int)blockIdx.x % C, inst = (int)blockIdx.x / C;
    const int nb = GRID ? q.n_bc_total : sp.inst[inst].n_bc, b0 = GRID ? 0 : sp.inst[inst].bc_first;
    const int N = (int)p.n, tid = threadIdx.x;
    const bool owner = rank < nb;
    const int b = b0 + rank;
    const long long first = *p.step + 1;  // t_n of the first step of the launch

    // cells of this block and their pull tables
    int n_cells, cell0 = 0;
    if (owner) {
        for (int k = tid; k < (int)(sizeof(BcParam) / 4); k += THREADS)
            reinterpret_cast<int *>(&s_P)[k] = reinterpret_cast<const int *>(q.par + b)[k];
        __syncthreads();
        n_cells = s_P.n_xf;
    } else {
        const int lo = sp.bulk_off[inst], n = sp.bulk_off[GRID ? sp.n_inst : inst + 1] - lo, w = C - nb, k = rank - nb;
        const int per = (n + w - 1) / w;
        cell0 = lo + min(k * per, n);
        n_cells = lo + min((k + 1) * per, n) - cell0;
    }
    const R omega = omega_of<R>(p, !GRID ? inst : owner ? s_P.inst : 0);
    int *tab = reinterpret_cast<int *>(smem);       // [18][n_cells]
    int *cell = tab + PULLS * n_cells;              // [n_cells]
    FirstLayer<R> *xf = reinterpret_cast<FirstLayer<R> *>((reinterpret_cast<uintptr_t>(cell + n_cells) + 15) & ~(uintptr_t)15);
    R *om = reinterpret_cast<R *>(xf);                // bulk of a grid: 1/tau of each cell
    FirstLayer<R> *v0s = xf + (owner ? n_cells : 0);  // closure velocities
    int2 *link = reinterpret_cast<int2 *>(v0s + (owner ? n_cells : 0));
    double *prof = reinterpret_cast<double *>(link + (owner ? s_P.n_links : 0));  // velocity inlet: 3 per node
    const int n_prof = owner && s_P.kind == BC_VELOCITY ? s_P.n_nodes : 0;
    R *unode = reinterpret_cast<R *>(prof + 3 * n_prof);
    for (int k = tid; k < n_cells; k += THREADS) {
        const int c = owner ? q.xf[s_P.xf_off + k] : sp.bulk[cell0 + k];
        cell[k] = c;
        pull_offsets(p, c, p.flags[c], tab + k, n_cells);
        if (GRID && !owner) om[k] = omega_of<R>(p, p.rows[find_row(p, c)].inst);
        if (owner) {
            const double *v0 = q.v0 + 3 * (size_t)(s_P.xf_off + k);
            v0s[k] = FirstLayer<R>{{(R)v0[0], (R)v0[1], (R)v0[2]}, R(0)};
        }
    }
    if (owner) {
        for (int k = tid; k < 3 * n_prof; k += THREADS) prof[k] = q.profile[3 * (size_t)s_P.node_off + k];
        for (int L = tid; L < s_P.n_links; L += THREADS) {
            const int g = s_P.link_off + L, i = q.lk_i[g];
            link[L] = make_int2(i * N + q.lk_xb[g], i | (q.lk_xfi[g] << 5) | (q.lk_node[g] << 16));
        }
        if (tid == 0) {
            s_st = q.state[(size_t)(first & 1) * q.n_bc_total + b];
            s_area = (double)s_P.n_xf;
            s_inv_area = 1.0 / s_area;
            s_third = (double)s_P.n_xf / 3.0;
            s_euler = boundary_euler(s_P);
        }
    }
    __syncthreads();
    const bool io_in = owner && sp.io_params && b == sp.io_b;
    const bool io_out = owner && sp.io_states && b >= sp.io_b0 && b < sp.io_b0 + sp.io_nb;

    // Threads of a boundary block: the first WORK collide its first layer and write
    // the ghosts; the next PREP prepare step s while those finish step s - 1 and
    // collide: its params (io), and the parts of its 0D model that do not depend
    // on its flow; the last warp stores states and waveforms.
    constexpr int AHEAD = THREADS / 4, WORK = THREADS - AHEAD, LAYER = WORK / BC_CHUNK * BC_CHUNK, PREP = AHEAD - 32;
    const int ta = tid - WORK;
    double given = 0.0;
    if (io_in && ta >= 0 && ta < sp.io_np) given = __ldcv(sp.io_params + ta);
    auto ahead = [&](int s) {
        const BcParam &P = s_P;
        const long long n = first + s;
        auto meet = [] { asm volatile("bar.sync 1, %0;" ::"n"(PREP) : "memory"); };
        if (io_in) {
            if (ta < sp.io_np) {
                s_P.par[ta] = given;
                sp.par[b].par[ta] = given;
                if (s + 1 < sp.n_steps) given = __ldcv(sp.io_params + (size_t)(s + 1) * sp.io_np + ta);
            }
            meet();
            if (ta == 0) s_euler = boundary_euler(P);
        }
        if (P.kind == BC_VELOCITY) {
            const double wt = P.par[0] * (double)(n + 1);
            if (ta == 0) s_cos = cos(wt);
            if (ta == 32) s_sin = sin(wt);
            meet();
            const double cosp = s_cos, sinp = s_sin;
            R *u = unode + (s & 1) * n_prof;  // the workers may still be reading step s - 1's
            for (int a = ta; a < n_prof; a += PREP) {  // the nodes' velocities at t_{n+1}
                const double *pr = prof + 3 * a;
                u[a] = (R)((double)P.sign * (pr[0] + pr[1] * cosp - pr[2] * sinp));
            }
        } else if (ta == 0) {
            ahead_terms(P, s_st, n, q.etab, &s_a);
        }
    };
    if (tid < NQ) {
        s_dir[tid][0] = c_ex[tid];
        s_dir[tid][1] = c_ey[tid];
        s_dir[tid][2] = c_ez[tid];
        s_dir[tid][3] = tid == 0 ? R(1.0 / 3.0) : (tid < 7 ? R(1.0 / 18.0) : R(1.0 / 36.0));
    }
    if (owner && ta >= 0 && ta < PREP) ahead(0);
    __syncthreads();

    const S *fin = f0;
    S *fout = f1;
    for (int s = 0; s < sp.n_steps; s++) {
        const OneBase<S> out{fout, N};
        const bool end = GRID && s + 1 == sp.n_steps;  // a grid needs no barrier after the last step
        if (!owner) {
            for (int k = tid; k < n_cells; k += THREADS) {
                const int c = cell[k];
                R f[NQ];
                f[0] = PlainLoad<S>::ld(fin + c);
#pragma unroll
                for (int i = 1; i < NQ; i++) f[i] = PlainLoad<S>::ld(fin + tab[(i - 1) * n_cells + k]);
                collide_store<S, R, false, false>(out, p, f, GRID ? om[k] : omega, 0u, c);
            }
            if (GRID) __syncthreads();
            __syncwarp();
            if (!end) barrier.arrive();
        } else {
            const BcParam &P = s_P;
            const long long n = first + s;
            for (int k0 = 0; k0 < P.n_red * BC_CHUNK; k0 += LAYER) {
                const int k = k0 + tid;
                double Q = 0.0, Ps = 0.0;
                if (tid < LAYER && k < n_cells) {
                    const int c = cell[k];
                    R f[NQ];
                    f[0] = PlainLoad<S>::ld(fin + c);
#pragma unroll
                    for (int i = 1; i < NQ; i++) f[i] = PlainLoad<S>::ld(fin + tab[(i - 1) * n_cells + k]);
                    const Moments<R> m = collide_store<S, R, false, false>(out, p, f, omega, 0u, c);
                    const R j = P.axis == 0 ? m.jx : P.axis == 1 ? m.jy : m.jz;
                    const R third = third_of(m.sd);
                    Q = (double)((R)P.sign * j / (R(1) + m.sd));
                    Ps = (double)third;
                    xf[k] = FirstLayer<R>{{m.jx, m.jy, m.jz}, third};
                }
                if (tid < LAYER) {
                    sQ[tid] = Q;
                    sP[tid] = Ps;
                }
                __syncthreads();
                // one warp per quantity and chunk of 256 cells.  The populations the
                // other blocks wait for are stored: a warp arrives at the cluster
                // barrier, which holds it until its stores are out, once the sums
                // and the 0D step no longer wait for it
                constexpr int CH = LAYER / BC_CHUNK;
                const int w = tid >> 5, h = w < CH ? w : w - CH, ch = k0 / BC_CHUNK + h;
                const bool last = k0 + LAYER >= P.n_red * BC_CHUNK;
                if (w < 2 * CH && ch < P.n_red) {
                    const double a = tree_256((w < CH ? sQ : sP) + h * BC_CHUNK);
                    if ((tid & 31) == 0) s_part[2 * ch + (w < CH ? 0 : 1)] = a;
                }
                __syncwarp();
                if (!GRID && last && w >= 2 * CH) barrier.arrive();
                __syncthreads();
                if (last && (GRID || (w > 0 && w < 2 * CH)) && !end) barrier.arrive();
            }
            // the thread's first two links (from the second warp on), their
            // populations in flight beside the 0D step
            constexpr int LINKS = WORK - 32;
            const int tl = tid - 32;
            int2 lk0 = make_int2(0, 0), lk1 = lk0;
            R post0 = R(0), post1 = R(0);
            auto post_of = [&](const int2 &lk) {
                return PlainLoad<S>::ld(fout + ((lk.y & 31) * N + cell[(lk.y >> 5) & 0x7ff]));
            };
            if (tl >= 0 && tid < WORK && tl < P.n_links) {
                lk0 = link[tl];
                post0 = post_of(lk0);
            }
            if (tl >= 0 && tid < WORK && tl + LINKS < P.n_links) {
                lk1 = link[tl + LINKS];
                post1 = post_of(lk1);
            }
            if (tid < 32) {
                const double a = sum_partials_pair(s_part, P.n_red);
                const double mean = quotient((tid & 1) ? s_third + a : a, s_area, s_inv_area);
                const double Ps = __shfl_sync(0xffffffffu, a, 1), Pbar = __shfl_sync(0xffffffffu, mean, 1);
                if (tid == 0) {
                    BcStepResult r;
                    const BcState old = s_st;
                    const BcState st =
                        s_euler ? zero_d_euler(P, old, s_a, a, mean, Pbar, n, &r.ptype, &r.closed, &r.S)
                                : zero_d_step(P, old, a, s_third + Ps, s_area, n, q.etab, &r.ptype, &r.closed, &r.S);
                    r.Pg = st.Pstar_gauge;
                    s_r = r;
                    s_st = st;
                }
            }
            __syncthreads();
            if (!GRID && tid < 32) barrier.arrive();
            if (tid < WORK) {
                const BcStepResult &r = s_r;
                const bool closed = r.closed != 0, ptype = r.ptype != 0;
                const R Pg = (R)r.Pg, Sm = (R)r.S;
                for (int L = tl >= 0 ? tl : P.n_links; L < P.n_links; L += LINKS) {
                    const int2 lk = L == tl ? lk0 : L == tl + LINKS ? lk1 : link[L];
                    const int i = lk.y & 31, xfi = (lk.y >> 5) & 0x7ff;
                    const FirstLayer<R> m = xf[xfi];
                    const R post = L == tl ? post0 : L == tl + LINKS ? post1 : post_of(lk);
                    R dP = R(0), vs[3] = {R(0), R(0), R(0)};
                    if (ptype) {
                        dP = Pg - m.p;
                        vs[0] = m.v[0];
                        vs[1] = m.v[1];
                        vs[2] = m.v[2];
                    } else if (P.kind == BC_VELOCITY) {
                        vs[P.axis] = unode[(s & 1) * n_prof + (lk.y >> 16)];
                    } else if (P.kind == BC_LV) {  // v_0(T_d) S(t, T_d, N_S); closing now, v_0 = v(x_f, T_d)
                        const FirstLayer<R> &u = closed ? xf[xfi] : v0s[xfi];
                        vs[0] = u.v[0] * Sm;
                        vs[1] = u.v[1] * Sm;
                        vs[2] = u.v[2] * Sm;
                    }
                    Storage<S>::st(fout + lk.x, post + feq_change<R>(s_dir[i][0], s_dir[i][1], s_dir[i][2], s_dir[i][3], dP, vs, m.v));
                }
                // the ghosts are pulled, and xf rewritten, by these threads only
                asm volatile("bar.sync 2, %0;" ::"n"(WORK) : "memory");
                if (closed && P.kind == BC_LV) {
                    for (int k = tid; k < n_cells; k += WORK) {
                        double *v0 = q.v0 + 3 * (size_t)(P.xf_off + k);
                        v0s[k] = xf[k];
                        for (int a = 0; a < 3; a++) v0[a] = (double)xf[k].v[a];
                    }
                    asm volatile("bar.sync 2, %0;" ::"n"(WORK) : "memory");
                }
            } else if (ta < PREP) {
                if (s + 1 < sp.n_steps) ahead(s + 1);
            } else {
                if (ta == PREP) {  // the state of t_{n+1} and the waveform row, as bc_step stores them
                    const BcState st = s_st;
                    q.state[(size_t)((n + 1) & 1) * q.n_bc_total + b] = st;
                    double *wv = q.wave + ((size_t)(n % q.wave_cap) * q.n_bc_total + b) * 4;
                    wv[0] = st.Qu;
                    wv[1] = st.Pbar - 1.0 / 3.0;
                    wv[2] = (P.kind == BC_RCR) ? st.Pw : (P.kind == BC_LV ? st.Pv : st.Pstar_gauge);
                    wv[3] = st.valve_open;
                    if (io_out)
                        state_row(st, P, q.etab, n + 1, sp.io_states + 8 * ((size_t)s * sp.io_nb + (b - sp.io_b0)));
                }
            }
        }
        const S *t = fin;
        fin = fout;
        fout = const_cast<S *>(t);
        __syncwarp();
        if (!end && !barrier.wait()) break;  // the other blocks' populations of this step are visible
    }
    // the last block to finish advances the step counter (all have read it; in a
    // grid, none still polls)
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(sp.done, 1) == (int)gridDim.x - 1) {
            *sp.done = 0;
            if (GRID) *sp.meet = 0u;
            *p.step = first + sp.n_steps - 1;
        }
    }
}

namespace {

template <class S> constexpr int small_threads() { return sizeof(typename Storage<S>::R) == 8 ? 512 : 1024; }

// cluster blocks per instance, or (cluster = 0) one cooperative grid
template <class S>
cudaLaunchConfig_t config(int cluster, int blocks, size_t smem, cudaStream_t st, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg{};
    if (cluster) {
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim = {(unsigned)cluster, 1, 1};
    } else {
        at->id = cudaLaunchAttributeCooperative;
        at->val.cooperative = 1;
    }
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(small_threads<S>());
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

template <class S> cudaError_t prepare(int cluster, size_t smem, int *at_once) {
    const auto k = cluster ? k_small_steps<S, small_threads<S>(), false> : k_small_steps<S, small_threads<S>(), true>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_MAX_SMEM);
    if (e == cudaSuccess && cluster > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    if (!cluster) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(at_once, k, small_threads<S>(), smem);
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = config<S>(cluster, cluster, smem, nullptr, &at);
    return cudaOccupancyMaxActiveClusters(at_once, k, &cfg);
}

template <class S> cudaError_t launch(void *f0, void *f1, const KParams &p, const BcKParams &q, const SmallKParams &sp,
                                      int blocks, size_t smem, cudaStream_t st) {
    const auto k = sp.cluster ? k_small_steps<S, small_threads<S>(), false> : k_small_steps<S, small_threads<S>(), true>;
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = config<S>(sp.cluster, blocks, smem, st, &at);
    return cudaLaunchKernelEx(&cfg, k, static_cast<S *>(f0), static_cast<S *>(f1), p, q, sp);
}

}  // namespace

cudaError_t prepare_small(int prec, int cluster, size_t smem, int *at_once) {
    cudaError_t e = cudaSuccess;
    DISPATCH(prec, e = prepare<S>(cluster, smem, at_once));
    return e;
}

cudaError_t launch_small(int prec, void *f0, void *f1, const KParams &p, const BcKParams &q, const SmallKParams &sp,
                         int blocks, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    DISPATCH(prec, e = launch<S>(f0, f1, p, q, sp, blocks, smem, st));
    return e;
}

}  // namespace lbm

// Device kernels of the per-step hot path besides the fused stream-collide
// (lbm_stream_collide.cu) and the immersed boundary (lbm_ib.cu):
//   k_bc_reduce       deterministic FP64 partial sums of the boundary flow Q
//                     and gauge pressure over the first fluid layer of each
//                     0D boundary (per-cell terms in the compute type), then,
//                     once per boundary, the FP64 forward-Euler 0D step (Eqs.
//                     rightbc, rightQ, LVE; valve switch and smoothing of
//                     Section 2.2.1)
//   k_bc_apply        the ghost populations of Eq. Non-equilibrium3 (per
//                     link, in the compute type)
//   k_boundary        both in one launch, a cluster of blocks per boundary
//   k_gather          read-out of f(t_n), P and j for the host
//   k_fields_box      FP32 read-out of P and j into box-order device arrays
//   k_wall_shear      wall shear stress at the fluid cells next to rigid walls
//   k_init, k_init_eq inverse of the pull: lays out a given f(t_0), or the
//                     equilibrium of given macroscopic fields
//   k_cycle_change    cycle-to-cycle change of the 0D waveforms
//
// Populations are stored as deviations s_i = f_i - w_i (FP32, FP16, BF16 or
// FP64) in structure-of-arrays order f[i][cell].  The resident state between
// steps is the post-collision field f*(t_n) with the ghost populations of
// the 0D boundary nodes for t_{n+1} already in their slots, so one step is:
// (immersed boundary) -> k_stream_collide -> k_bc_reduce -> k_bc_apply.
#include <cooperative_groups.h>

#include "lbm_ghost.cuh"
#include "lbm_device.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// 0D coupling.  The per-cell and per-link arithmetic runs in the compute type
// R of the populations (FP32 for FP32/FP16/BF16 storage: the FP64 pipe of
// this part is narrow), with pressures as deviations from P_ref = 1/3 so that
// FP32 keeps their resolution; the boundary sums and the 0D step are FP64.
template <class R>
__device__ __forceinline__ void forced_velocity(const KParams &p, int cf, R v[3]) {
    const size_t N = (size_t)p.n;
    const R *aux = static_cast<const R *>(p.aux);
    v[0] = aux[N + cf];
    v[1] = aux[2 * N + cf];
    v[2] = aux[3 * N + cf];
    if (__ldg(&p.flags[cf]) & FL_BAND) {
        const typename Vec4<R>::T bb = static_cast<const typename Vec4<R>::T *>(p.b)[cf];
        v[0] += R(0.5) * bb.x;
        v[1] += R(0.5) * bb.y;
        v[2] += R(0.5) * bb.z;
    }
}

// The boundary's partial sums added by one warp in a fixed order (lane k
// takes partials k, k + 32, ..., then a butterfly), so that every caller gets
// the same bits.
static __device__ __forceinline__ void bc_sum_partials(const BcParam &P, const BcKParams &q, double *Q, double *Ps) {
    const int lane = threadIdx.x & 31;
    double a = 0.0, c = 0.0;
    for (int k = lane; k < P.n_red; k += 32) {
        a += __ldcg(&q.partial[2 * (P.red_off + k)]);
        c += __ldcg(&q.partial[2 * (P.red_off + k) + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    *Q = a;
    *Ps = c;
}

// Partial sums of the boundary flow Q = sum n.j / sum f and of the gauge
// pressure (P - P_ref = c_s^2 sum s) over one chunk of a boundary's first
// fluid layer (FP64 sums in a fixed tree order).  With q.step_in_reduce (many
// link blocks), the boundary's last chunk to arrive (a counter per boundary;
// no block waits for another) sums all partials and takes the 0D step once
// for the boundary; otherwise every link block of k_bc_apply takes it.
template <class R>
__global__ void __launch_bounds__(BC_CHUNK) k_bc_reduce(KParams p, BcKParams q) {
    const int b = q.red_bc[blockIdx.x], ch = q.red_chunk[blockIdx.x];
    const BcParam &P = q.par[b];
    const size_t N = (size_t)p.n;
    const R *aux = static_cast<const R *>(p.aux);
    const int a = ch * BC_CHUNK + threadIdx.x;
    __shared__ double sQ[BC_CHUNK], sP[BC_CHUNK];
    __shared__ int s_last;
    double Q = 0.0, Ps = 0.0;
    if (a < P.n_xf) {
        const int cf = q.xf[P.xf_off + a];
        const R sd = aux[cf];
        Q = (double)((R)P.sign * aux[(size_t)(1 + P.axis) * N + cf] / (R(1) + sd));
        Ps = (double)(sd / R(3));
    }
    sQ[threadIdx.x] = Q;
    sP[threadIdx.x] = Ps;
    __syncthreads();
    for (int s = BC_CHUNK / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sQ[threadIdx.x] += sQ[threadIdx.x + s];
            sP[threadIdx.x] += sP[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        q.partial[2 * (P.red_off + ch)] = sQ[0];
        q.partial[2 * (P.red_off + ch) + 1] = sP[0];
        if (q.step_in_reduce) {
            __threadfence();  // the partial is visible before the arrival is counted
            s_last = atomicAdd(&q.arrived[b], 1) == P.n_red - 1;
        }
    }
    if (!q.step_in_reduce) return;
    __syncthreads();
    if (!s_last || threadIdx.x >= 32) return;
    __threadfence();
    bc_sum_partials(P, q, &Q, &Ps);
    if (threadIdx.x != 0) return;
    q.arrived[b] = 0;  // for the next step (kernel boundaries order it)
    q.result[b] = bc_step(P, b, Q, Ps, *p.step, q, true);
}

// Ghost populations of one chunk of links, Eq. Non-equilibrium3 written as
//   f_i(x_b) = f*_i(x_f) + f^eq_i(P*, v*) - f^eq_i(P(x_f), v(x_f)),
// since f*_i(x_f) = f^eq_i + (1 - 1/tau) f^neq_i + F_i at x_f.
// STEP_HERE: the kernel for few link blocks, each of which takes the 0D step
// itself (the boundary's first chunk storing the state); otherwise the step's
// result comes from k_bc_reduce.  Two instances, so that the one without the
// step keeps its low register count.
template <class S, bool STEP_HERE>
__global__ void __launch_bounds__(BC_CHUNK) k_bc_apply(S *__restrict__ f, KParams p, BcKParams q) {
    using R = typename Storage<S>::R;
    const int b = q.app_bc[blockIdx.x], ch = q.app_chunk[blockIdx.x];
    const BcParam &P = q.par[b];
    const size_t N = (size_t)p.n;
    const R *aux = static_cast<const R *>(p.aux);
    const int L = ch * BC_CHUNK + threadIdx.x;
    const bool have = L < P.n_links;
    if (!STEP_HERE && !have) return;
    // the link's inputs, read before the 0D step's result is known (with
    // STEP_HERE they arrive while one thread takes the step): x_b, x_f and i,
    // the forced velocity, sum s and f*_i at x_f, and the closure velocity or
    // the inlet profile of the link's node
    int cb = 0, cf = 0, i = 0;
    R vf[3] = {R(0), R(0), R(0)}, sdf = R(0), post = R(0);
    double pr[3] = {0.0, 0.0, 0.0}, v0o[3] = {0.0, 0.0, 0.0};
    if (have) {
        cb = q.lk_xb[P.link_off + L];
        cf = q.lk_xf[P.link_off + L];
        i = q.lk_i[P.link_off + L];
        forced_velocity<R>(p, cf, vf);
        sdf = aux[cf];
        post = Storage<S>::ld(f + pidx(i, (uint32_t)cf, (uint32_t)N));
        if (P.kind == BC_VELOCITY) {
            const double *prof = q.profile + 3 * (size_t)(P.node_off + q.lk_node[P.link_off + L]);
            pr[0] = prof[0];
            pr[1] = prof[1];
            pr[2] = prof[2];
        } else if (P.kind == BC_LV) {  // v_0(T_d) of an earlier closure (rewritten below if one happens now)
            const double *v0 = q.v0 + 3 * (size_t)(P.xf_off + q.lk_xfi[P.link_off + L]);
            v0o[0] = v0[0];
            v0o[1] = v0[1];
            v0o[2] = v0[2];
        }
    }
    BcStepResult r;
    if (!STEP_HERE) {
        r = q.result[b];
    } else {
        __shared__ BcStepResult s_r;
        if (threadIdx.x < 32) {
            double Q, Ps;
            bc_sum_partials(P, q, &Q, &Ps);
            if (threadIdx.x == 0) s_r = bc_step(P, b, Q, Ps, *p.step, q, ch == 0);
        }
        __syncthreads();
        if (!have) return;
        r = s_r;
    }
    const R dfeq = ghost_change<R>(P, r, i, vf, sdf, pr, v0o,
                                   P.kind == BC_LV ? q.v0 + 3 * (size_t)(P.xf_off + q.lk_xfi[P.link_off + L]) : nullptr);
    Storage<S>::st(f + pidx(i, (uint32_t)cb, (uint32_t)N), post + dfeq);
}

// The whole boundary work of a step in one launch (lattices without wall nodes):
// one cluster of blocks per boundary.  The blocks sum their chunks of 256
// first-layer cells (the tree of k_bc_reduce); after a cluster barrier the
// first block adds the partials, takes the 0D step and hands the result to the
// others' shared memory; after another every block writes its links' ghosts,
// whose inputs it has read beside all this.  Per-step 0D input and output
// (lbm_step_io) is part of it: the params come straight from the host's memory
// while the sums run, the state rows go there after the ghosts.  Same
// expressions and orders as k_bc_reduce and k_bc_apply, the same bits.
// Bound by latency (two cluster barriers, the trees, FP64 divisions of 700
// cycles).  One launch and its start hidden behind stream-collide's end: tube
// of 172k cells 14.5 -> 12.4 us per step (FP16 14.2 -> 12.4), 20.1 -> 14.6 with
// per-step 0D input and output (three launches and two of one warp before),
// 64 tubes of 14k cells 36.6 -> 30.1.  A boundary of more links than its blocks
// have threads (12.5 -> 13.0 us at 6,100 links), FP64 (whose ghosts need the FP64
// pipes of many SMs: 25 -> 33 us) and batches with more clusters than SMs
// take at once (96 uneven tubes 528 -> 617 us) keep the two kernels: beyond 300
// blocks, of 512 threads, one of which fills an SM's registers, beyond 200 (tubes of
// 108,540 cells, 16 blocks each, two kernels -> one: 4 18.3 -> 15.7 us per step, 10 36.5 ->
// 34.3, 12 40.0 -> 39.6, 14 44.6 -> 45.9, 18 53.2 -> 58.5; FP16 10 27.0 -> 25.2, 14 34.5 -> 40.1, 18
// 42.3 -> 48.3).
template <class S, int BS>
__global__ void __launch_bounds__(BS) k_boundary(S *__restrict__ f, KParams p, BcKParams q, BcIo io) {
    using R = typename Storage<S>::R;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double sQ[BS], sP[BS], s_area, s_inv_area, s_third, s_cos, s_sin;
    __shared__ BcParam s_P;
    __shared__ BcState s_st;
    __shared__ BcStepResult s_r;
    __shared__ Ahead s_a;
    __shared__ int s_euler;
    cluster.barrier_arrive();  // waited for before the first block writes into the others
    let_next_start();
    const int CL = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), b = q.bc0 + blockIdx.x / CL;
    const int tid = threadIdx.x;
    const size_t N = (size_t)p.n;
    const R *aux = static_cast<const R *>(p.aux);
    for (int k = tid; k < (int)(sizeof(BcParam) / 4); k += BS)
        reinterpret_cast<int *>(&s_P)[k] = reinterpret_cast<const int *>(q.par + b)[k];
    wait_for_previous();  // stream-collide of this step
    const long long n = *p.step;
    const bool io_in = rank == 0 && io.params && b == io.b;
    __syncthreads();
    if (io_in && tid < io.np) {
        const double v = __ldcv(io.params + (n - *io.base) * io.np + tid);
        s_P.par[tid] = v;
        io.par[b].par[tid] = v;
    }
    if (io_in) __syncthreads();
    const BcParam &P = s_P;
    // the thread's first link: read before the sums, used after the 0D step
    struct Link {
        int cb, cf, i;
        R vf[3], sd, post;
        double pr[3], v0[3];
    };
    auto load_link = [&](int L, Link &k) {
        k.cb = q.lk_xb[P.link_off + L];
        k.cf = q.lk_xf[P.link_off + L];
        k.i = q.lk_i[P.link_off + L];
        forced_velocity<R>(p, k.cf, k.vf);
        k.sd = aux[k.cf];
        k.post = Storage<S>::ld(f + pidx(k.i, (uint32_t)k.cf, (uint32_t)N));
        if (P.kind == BC_VELOCITY) {
            const double *prof = q.profile + 3 * (size_t)(P.node_off + q.lk_node[P.link_off + L]);
            k.pr[0] = prof[0];
            k.pr[1] = prof[1];
            k.pr[2] = prof[2];
        } else if (P.kind == BC_LV) {
            const double *v0 = q.v0 + 3 * (size_t)(P.xf_off + q.lk_xfi[P.link_off + L]);
            k.v0[0] = v0[0];
            k.v0[1] = v0[1];
            k.v0[2] = v0[2];
        }
    };
    const int L0 = rank * BS + tid;
    Link first;
    if (L0 < P.n_links) load_link(L0, first);
    if (rank == 0) {  // beside the sums, on warps of their own
        if (P.kind == BC_VELOCITY) {
            const double wt = P.par[0] * (double)(n + 1);
            if (tid == BS - 32) s_cos = cos(wt);
            if (tid == BS - 64) s_sin = sin(wt);
        } else if (tid == BS - 32) {
            const BcState st = q.state[(size_t)(n & 1) * q.n_bc_total + b];
            ahead_terms(P, st, n, q.etab, &s_a);
        }
        if (tid == BS - 96) s_st = q.state[(size_t)(n & 1) * q.n_bc_total + b];
        if (tid == BS - 128) {
            s_area = (double)P.n_xf;
            s_inv_area = 1.0 / s_area;
            s_third = s_area / 3.0;
            s_euler = boundary_euler(P);
        }
    }
    for (int k0 = rank * BS; k0 < P.n_red * BC_CHUNK; k0 += CL * BS) {
        const int a = k0 + tid;
        double Q = 0.0, Ps = 0.0;
        if (a < P.n_xf) {
            const int cf = q.xf[P.xf_off + a];
            const R sd = aux[cf];
            Q = (double)((R)P.sign * aux[(size_t)(1 + P.axis) * N + cf] / (R(1) + sd));
            Ps = (double)(sd / R(3));
        }
        sQ[tid] = Q;
        sP[tid] = Ps;
        __syncthreads();
        constexpr int CH = BS / BC_CHUNK;
        const int w = tid >> 5, ch = k0 / BC_CHUNK + (w & (CH - 1));
        if (w < 2 * CH && ch < P.n_red) {  // one warp per quantity and chunk
            const double t = tree_256((w < CH ? sQ : sP) + (w & (CH - 1)) * BC_CHUNK);
            if ((tid & 31) == 0) q.partial[2 * (P.red_off + ch) + (w < CH ? 0 : 1)] = t;
        }
        __syncthreads();
    }
    __syncwarp();
    cluster.barrier_wait();
    cluster.sync();  // the partials are visible to the cluster
    if (rank == 0) {
        if (tid < 32) {
            const double a = sum_partials_pair(q.partial + 2 * P.red_off, P.n_red);
            const double mean = quotient((tid & 1) ? s_third + a : a, s_area, s_inv_area);
            const double Ps = __shfl_sync(0xffffffffu, a, 1), Pbar = __shfl_sync(0xffffffffu, mean, 1);
            if (tid == 0) {
                BcStepResult r;
                const BcState old = s_st;
                s_st = s_euler ? zero_d_euler(P, old, s_a, a, mean, Pbar, n, &r.ptype, &r.closed, &r.S)
                               : zero_d_step(P, old, a, s_third + Ps, s_area, n, q.etab, &r.ptype, &r.closed, &r.S);
                r.Pg = s_st.Pstar_gauge;
                r.cosp = s_cos;
                r.sinp = s_sin;
                r.pad0 = r.pad1 = 0;
                s_r = r;
            }
            __syncwarp();
            constexpr int W = (int)(sizeof(BcStepResult) / 8);
            for (int k = tid; k < W * (CL - 1); k += 32)
                reinterpret_cast<unsigned long long *>(cluster.map_shared_rank(&s_r, 1 + k / W))[k % W] =
                    reinterpret_cast<const unsigned long long *>(&s_r)[k % W];
        }
    }
    __syncwarp();
    cluster.sync();  // the result is in every block's shared memory
    const BcStepResult r = s_r;
    for (int L = L0; L < P.n_links; L += CL * BS) {
        if (L != L0) load_link(L, first);
        const R d = ghost_change<R>(P, r, first.i, first.vf, first.sd, first.pr, first.v0,
                                    P.kind == BC_LV ? q.v0 + 3 * (size_t)(P.xf_off + q.lk_xfi[P.link_off + L]) : nullptr);
        Storage<S>::st(f + pidx(first.i, (uint32_t)first.cb, (uint32_t)N), first.post + d);
    }
    if (rank == 0 && tid == BS - 32) {  // the state of t_{n+1} and the waveform row, as bc_step stores them
        const BcState st = s_st;
        q.state[(size_t)((n + 1) & 1) * q.n_bc_total + b] = st;
        double *w = q.wave + ((size_t)(n % q.wave_cap) * q.n_bc_total + b) * 4;
        w[0] = st.Qu;
        w[1] = st.Pbar - 1.0 / 3.0;
        w[2] = (P.kind == BC_RCR) ? st.Pw : (P.kind == BC_LV ? st.Pv : st.Pstar_gauge);
        w[3] = st.valve_open;
        if (io.states && b >= io.b0 && b < io.b0 + io.nb)
            state_row(st, P, q.etab, n + 1, io.states + 8 * ((size_t)(n - *io.base) * io.nb + (b - io.b0)));
    }
}

// ---------------------------------------------------------------------------
// Read-out: f(t_n) = pull of the resident f*(t_{n-1}) (with ghosts), plus
// P = c_s^2 sum f and j = sum e f, for the cells [c0, c1) of one instance
// (outputs indexed c - c0 with stride M = c1 - c0; non-fluid cells get 0).
template <class S>
__global__ void k_gather(const S *__restrict__ fin, KParams p, int c0, int c1, double *fout19, double *mac4) {
    const int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= c1) return;
    const uint32_t fl = p.flags[c];
    const size_t N = (size_t)p.n, M = (size_t)(c1 - c0), k = (size_t)(c - c0);
    if (!(fl & FL_ACTIVE)) {
        if (fout19)
            for (int i = 0; i < NQ; i++) fout19[i * M + k] = 0.0;
        for (int a = 0; a < 4; a++) mac4[a * M + k] = 0.0;
        return;
    }
    const int r = find_row(p, c);
    const int x = p.rows[r].x0 + (c - p.rows[r].off);
    double sum = 0, jx = 0, jy = 0, jz = 0;
    for (int i = 0; i < NQ; i++) {
        size_t idx;
        if (i == 0) idx = pidx(0, (uint32_t)c, (uint32_t)N);
        else if (fl & (1u << i)) idx = pidx(opp(i), (uint32_t)c, (uint32_t)N);
        else idx = pidx(i, (uint32_t)(p.rows[r].nb[nbk(i)] + x - cx(i)), (uint32_t)N);
        const double fi = (double)Storage<S>::ld(fin + idx) + wgt(i);
        if (fout19) fout19[i * M + k] = fi;
        sum += fi;
        jx += cx(i) * fi;
        jy += cy(i) * fi;
        jz += cz(i) * fi;
    }
    mac4[k] = sum / 3.0;
    mac4[M + k] = jx;
    mac4[2 * M + k] = jy;
    mac4[3 * M + k] = jz;
}

// Inverse of the pull: given f(t_0) at the fluid cells of [c0, c1), write
// every population into the slot it will be pulled from.
template <class S>
__global__ void k_init(S *__restrict__ fout, KParams p, const double *__restrict__ f19, int c0, int c1) {
    const int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= c1) return;
    const uint32_t fl = p.flags[c];
    if (!(fl & FL_ACTIVE)) return;
    const size_t N = (size_t)p.n;
    const size_t M = (size_t)(c1 - c0);
    const int r = find_row(p, c);
    const int x = p.rows[r].x0 + (c - p.rows[r].off);
    for (int i = 0; i < NQ; i++) {
        const double s = f19[i * M + (c - c0)] - wgt(i);
        size_t idx;
        if (i == 0) idx = pidx(0, (uint32_t)c, (uint32_t)N);
        else if (fl & (1u << i)) idx = pidx(opp(i), (uint32_t)c, (uint32_t)N);
        else idx = pidx(i, (uint32_t)(p.rows[r].nb[nbk(i)] + x - cx(i)), (uint32_t)N);
        Storage<S>::st(fout + idx, (typename Storage<S>::R)s);
    }
}

// Wall shear stress at the fluid cells next to a rigid wall (the paper's
// case-study observable, WSS = mu dv_1/dx_3 there): viscous stress of f(t_n)
// from its non-equilibrium part, sigma = -(1 - 1/(2 tau)) [sum_i e_i e_i
// (f_i - f^eq_i) + (v b + b v)/2], traction on the wall normal n (the
// normalised sum of e_i over bounce-back directions, into the fluid), minus
// its normal part.  Output 3 doubles per cell of [c0, c1) (zero elsewhere).
template <class S>
__global__ void k_wall_shear(const S *__restrict__ fin, KParams p, int c0, int c1, double *out3) {
    const int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= c1) return;
    const size_t N = (size_t)p.n, M = (size_t)(c1 - c0), k = (size_t)(c - c0);
    const uint32_t fl = p.flags[c];
    out3[k] = out3[M + k] = out3[2 * M + k] = 0.0;
    if (!(fl & FL_ACTIVE) || !(fl & FL_BBMASK)) return;
    const int r = find_row(p, c);
    const int x = p.rows[r].x0 + (c - p.rows[r].off);
    double f[NQ], sum = 0, jx = 0, jy = 0, jz = 0, n[3] = {0, 0, 0};
    for (int i = 0; i < NQ; i++) {
        size_t idx;
        if (i == 0) idx = pidx(0, (uint32_t)c, (uint32_t)N);
        else if (fl & (1u << i)) idx = pidx(opp(i), (uint32_t)c, (uint32_t)N);
        else idx = pidx(i, (uint32_t)(p.rows[r].nb[nbk(i)] + x - cx(i)), (uint32_t)N);
        f[i] = (double)Storage<S>::ld(fin + idx) + wgt(i);
        sum += f[i];
        jx += cx(i) * f[i];
        jy += cy(i) * f[i];
        jz += cz(i) * f[i];
        if (i > 0 && (fl & (1u << i))) {
            n[0] += cx(i);
            n[1] += cy(i);
            n[2] += cz(i);
        }
    }
    const double nn = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    if (nn == 0.0) return;
    n[0] /= nn;
    n[1] /= nn;
    n[2] /= nn;
    double b[3] = {0, 0, 0};
    if (fl & FL_BAND) {
        using R = typename Storage<S>::R;
        const typename Vec4<R>::T bb = static_cast<const typename Vec4<R>::T *>(p.b)[c];
        b[0] = bb.x;
        b[1] = bb.y;
        b[2] = bb.z;
    }
    const double v[3] = {jx + 0.5 * b[0], jy + 0.5 * b[1], jz + 0.5 * b[2]};
    const double P = sum / 3.0, usq = 1.5 * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    double pi[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    for (int i = 0; i < NQ; i++) {
        const double e[3] = {(double)cx(i), (double)cy(i), (double)cz(i)};
        const double eu = e[0] * v[0] + e[1] * v[1] + e[2] * v[2];
        const double fneq = f[i] - wgt(i) * (3.0 * P + 3.0 * eu + 4.5 * eu * eu - usq);
        for (int a = 0; a < 3; a++)
            for (int q = 0; q < 3; q++) pi[a][q] += e[a] * e[q] * fneq;
    }
    const double kf = -(1.0 - 0.5 * p.omega[p.rows[r].inst]);
    double t[3], tn = 0.0;
    for (int a = 0; a < 3; a++) {
        t[a] = 0.0;
        for (int q = 0; q < 3; q++) t[a] += kf * (pi[a][q] + 0.5 * (v[a] * b[q] + b[a] * v[q])) * n[q];
        tn += t[a] * n[a];
    }
    for (int a = 0; a < 3; a++) out3[a * M + k] = t[a] - tn * n[a];
}

// Equilibrium initialisation: f_i(x, t_0) = f^eq_i(P, v) (Eq. feq) from the
// macroscopic fields of the fluid cells of [c0, c1) (4 x M doubles: P, vx,
// vy, vz), laid out by the inverse of the pull like k_init.
template <class S>
__global__ void k_init_eq(S *__restrict__ fout, KParams p, const double *__restrict__ mac, int c0, int c1) {
    const int c = c0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= c1) return;
    const uint32_t fl = p.flags[c];
    if (!(fl & FL_ACTIVE)) return;
    const size_t N = (size_t)p.n, M = (size_t)(c1 - c0), k = (size_t)(c - c0);
    const double P = mac[k], vx = mac[M + k], vy = mac[2 * M + k], vz = mac[3 * M + k];
    const double usq = 1.5 * (vx * vx + vy * vy + vz * vz);
    const int r = find_row(p, c);
    const int x = p.rows[r].x0 + (c - p.rows[r].off);
    for (int i = 0; i < NQ; i++) {
        const double eu = cx(i) * vx + cy(i) * vy + cz(i) * vz;
        const double s = wgt(i) * (3.0 * P - 1.0 + 3.0 * eu + 4.5 * eu * eu - usq);  // f^eq_i - w_i
        size_t idx;
        if (i == 0) idx = pidx(0, (uint32_t)c, (uint32_t)N);
        else if (fl & (1u << i)) idx = pidx(opp(i), (uint32_t)c, (uint32_t)N);
        else idx = pidx(i, (uint32_t)(p.rows[r].nb[nbk(i)] + x - cx(i)), (uint32_t)N);
        Storage<S>::st(fout + idx, (typename Storage<S>::R)s);
    }
}

// Cycle-to-cycle change of the boundary waveforms of one instance per CTA:
// over the last `period` recorded steps t, max over waveforms W in {Q_u, mean
// P} of each boundary of max_t |W(t) - W(t - period)| / max_t |W(t - period)|.
__global__ void k_cycle_change(BcKParams q, const int *bc_first, const int *n_bc, const long long *period,
                               long long steps, double *delta) {
    const int inst = blockIdx.x;
    const long long T = period[inst];
    if (T <= 0) {
        if (threadIdx.x == 0) delta[inst] = -1.0;
        return;
    }
    __shared__ double s_num[256], s_den[256];
    double worst = 0.0;
    for (int k = 0; k < n_bc[inst]; k++) {
        const int b = bc_first[inst] + k;
        for (int wv = 0; wv < 2; wv++) {
            double num = 0.0, den = 0.0;
            for (long long t = steps - T + threadIdx.x; t < steps; t += blockDim.x) {
                const double a = q.wave[((size_t)(t % q.wave_cap) * q.n_bc_total + b) * 4 + wv];
                const double c = q.wave[((size_t)((t - T) % q.wave_cap) * q.n_bc_total + b) * 4 + wv];
                num = fmax(num, fabs(a - c));
                den = fmax(den, fabs(c));
            }
            s_num[threadIdx.x] = num;
            s_den[threadIdx.x] = den;
            __syncthreads();
            for (int s = blockDim.x / 2; s > 0; s >>= 1) {
                if (threadIdx.x < s) {
                    s_num[threadIdx.x] = fmax(s_num[threadIdx.x], s_num[threadIdx.x + s]);
                    s_den[threadIdx.x] = fmax(s_den[threadIdx.x], s_den[threadIdx.x + s]);
                }
                __syncthreads();
            }
            if (s_den[0] > 0.0) worst = fmax(worst, s_num[0] / s_den[0]);
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) delta[inst] = worst;
}

// ---------------------------------------------------------------------------
// launchers

template <class S, int BS>
static cudaError_t boundary_in_one(void *f, const KParams &p, const BcKParams &q, const BcIo &io, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[3] = {};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)q.cluster, 1, 1};
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_early
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(q.n_bc * q.cluster));
    cfg.blockDim = dim3(BS);
    cfg.stream = s;
    at[2].id = cudaLaunchAttributePriority;
    at[2].val.priority = q.priority;
    cfg.attrs = at;
    cfg.numAttrs = q.priority ? 3 : 2;
    return cudaLaunchKernelEx(&cfg, k_boundary<S, BS>, as<S>(f), p, q, io);
}

cudaError_t launch_boundary(int prec, void *f, const KParams &p, const BcKParams &q, const BcIo &io, cudaStream_t s) {
    if (q.n_bc == 0) return cudaSuccess;
    if (q.cluster) {  // never in FP64 (lbm_create)
        cudaError_t e = cudaSuccess;
        if (q.wide) {
            DISPATCH_F32(prec, (e = boundary_in_one<S, 512>(f, p, q, io, s)));
        } else {
            DISPATCH_F32(prec, (e = boundary_in_one<S, 256>(f, p, q, io, s)));
        }
        return e;
    }
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributePriority;
    at.val.priority = q.priority;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)q.n_red_blocks);
    cfg.blockDim = dim3(BC_CHUNK);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = q.priority ? 1 : 0;
    cudaError_t e = prec == 3 ? cudaLaunchKernelEx(&cfg, k_bc_reduce<double>, p, q)
                              : cudaLaunchKernelEx(&cfg, k_bc_reduce<float>, p, q);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3((unsigned)q.n_app_blocks);
    if (q.step_in_reduce) {
        DISPATCH(prec, (e = cudaLaunchKernelEx(&cfg, k_bc_apply<S, false>, as<S>(f), p, q)));
    } else {
        DISPATCH(prec, (e = cudaLaunchKernelEx(&cfg, k_bc_apply<S, true>, as<S>(f), p, q)));
    }
    return e;
}

cudaError_t launch_gather(int prec, const void *fin, const KParams &p, int c0, int c1, double *f19, double *mac4,
                          cudaStream_t s) {
    const int block = 256;
    const int grid = (c1 - c0 + block - 1) / block;
    if (grid == 0) return cudaSuccess;
    DISPATCH(prec, (k_gather<S><<<grid, block, 0, s>>>(static_cast<const S *>(fin), p, c0, c1, f19, mac4)));
    return cudaGetLastError();
}

// 0D state rows of boundaries [b0, b0 + nb) for lbm_read_0d_state_async
__global__ void k_state_rows(const BcState *__restrict__ st, const BcParam *__restrict__ par,
                             const double *__restrict__ etab, int b0, int nb, int nbc_total, long long steps,
                             double *out8) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nb) return;
    state_row(st[(size_t)(steps & 1) * nbc_total + b0 + k], par[b0 + k], etab, steps, out8 + 8 * (size_t)k);
}

// Per-step 0D input and output of lbm_step_io, in stream order around each
// step.  *cursor counts the call's steps taken so far.  k_io_params copies the
// np params of step *cursor (from page-locked host memory that the device
// addresses) into the boundary's device parameters; k_io_state writes the
// state rows of nb boundaries after the step (step count *step + 1, the step
// index t_n of the step just taken plus one) to out8 + 8 nb *cursor and then
// advances *cursor.
__global__ void k_io_params(const double *__restrict__ params, int np, BcParam *par, const long long *cursor) {
    const long long c = *cursor;
    if ((int)threadIdx.x < np) par->par[threadIdx.x] = params[c * np + threadIdx.x];
}

__global__ void k_io_state(const BcState *__restrict__ st, const BcParam *__restrict__ par,
                           const double *__restrict__ etab, int b0, int nb, int nbc_total,
                           const long long *__restrict__ step, double *out8, long long *cursor) {
    const long long c = *cursor;
    const int k = threadIdx.x;
    const long long steps = *step + 1;
    if (k < nb)
        state_row(st[(size_t)(steps & 1) * nbc_total + b0 + k], par[b0 + k], etab, steps,
                  out8 + 8 * ((size_t)c * nb + k));
    __syncthreads();
    if (threadIdx.x == 0) *cursor = c + 1;
}

// the step count after the steps so far: the first row of lbm_step_io's arrays
__global__ void k_io_base(const long long *step, long long *base) { *base = *step + 1; }

cudaError_t launch_io_base(const long long *step, long long *base, cudaStream_t s) {
    k_io_base<<<1, 1, 0, s>>>(step, base);
    return cudaGetLastError();
}

cudaError_t launch_io_params(const double *params, int np, BcParam *par, const long long *cursor, cudaStream_t s) {
    k_io_params<<<1, 32, 0, s>>>(params, np, par, cursor);
    return cudaGetLastError();
}

cudaError_t launch_io_state(const BcState *st, const BcParam *par, const double *etab, int b0, int nb, int nbc_total,
                            const long long *step, double *out8, long long *cursor, cudaStream_t s) {
    k_io_state<<<1, 32 * ((nb + 31) / 32), 0, s>>>(st, par, etab, b0, nb, nbc_total, step, out8, cursor);
    return cudaGetLastError();
}

cudaError_t launch_state_rows(const BcState *st, const BcParam *par, const double *etab, int b0, int nb,
                              int nbc_total, long long steps, double *out8, cudaStream_t s) {
    if (nb == 0) return cudaSuccess;
    k_state_rows<<<1, 32 * ((nb + 31) / 32), 0, s>>>(st, par, etab, b0, nb, nbc_total, steps, out8);
    return cudaGetLastError();
}

// Small stream-ordered transfer in 8-byte words, between mapped page-locked
// host memory and device memory, on the compute engine (no hand-off to a
// copy engine and back).
__global__ void k_copy_words(const unsigned long long *__restrict__ src, unsigned long long *__restrict__ dst,
                             int n) {
    for (int k = threadIdx.x; k < n; k += blockDim.x) dst[k] = src[k];
}

// the step counter, copied for each part of a step graph
__global__ void k_spread_step(const long long *step, long long *out, int n) {
    if ((int)threadIdx.x < n) out[threadIdx.x] = *step;
}

cudaError_t launch_spread_step(const long long *step, long long *out, int n, cudaStream_t s) {
    k_spread_step<<<1, 32, 0, s>>>(step, out, n);
    return cudaGetLastError();
}

cudaError_t launch_copy_words(const void *src, void *dst, size_t bytes, cudaStream_t s) {
    if (bytes == 0) return cudaSuccess;
    if (bytes % 8 != 0) return cudaErrorInvalidValue;
    k_copy_words<<<1, 32, 0, s>>>(static_cast<const unsigned long long *>(src), static_cast<unsigned long long *>(dst),
                                  (int)(bytes / 8));
    return cudaGetLastError();
}

// Sums of population deviations for the FP32 read-out, no less exact than FP64
// ones.  FP32 and BF16 storage adds in triples of FP32 (two two-sums and a plain
// sum, error about 2^-70 of the terms).  FP16 populations are multiples of 2^-24,
// so that pairs of FP32 (one two-sum) hold their sums exactly (below 2^14); of
// FP32 populations pairs lost 2^-46 of the terms, up to 25 times as much as FP64
// where the terms cancel over many binades.  FP64 storage adds in FP64.
template <bool TRIPLE> struct SplitSum {
    float h = 0.f, l = 0.f, c = 0.f;
    static __device__ __forceinline__ float two_sum(float &s, float x) {  // s += x; what the rounding left out
        const float a = s, t = a + x, d = t - a;
        s = t;
        return (a - (t - d)) + (x - d);
    }
    __device__ __forceinline__ void add(float x) {
        const float e = two_sum(h, x);
        if (TRIPLE) c += two_sum(l, e);
        else l += e;
    }
    // h + l + c as a leading part and the rest; an infinity or NaN in h makes l and
    // the rest NaNs: then h alone is the sum
    __device__ __forceinline__ float split(float *rest) const {
        float s = h;
        *rest = two_sum(s, l) + c;
        return s;
    }
    __device__ __forceinline__ float value() const {
        float r;
        const float s = split(&r);
        return isfinite(r) ? s + r : h;
    }
    __device__ __forceinline__ float pressure() const {  // (1 + h + l + c) / 3 to the last bit or so
        SplitSum t = *this;
        t.add(1.f);
        float r;
        const float s = t.split(&r), q = s * (1.f / 3.f);
        r = (fmaf(-3.f, q, s) + r) * (1.f / 3.f);
        return isfinite(r) ? q + r : t.h * (1.f / 3.f);
    }
};
struct WideSum {
    double h = 0.0;
    __device__ __forceinline__ void add(double x) { h += x; }
    __device__ __forceinline__ float value() const { return (float)h; }
    __device__ __forceinline__ float pressure() const { return (float)((1.0 + h) / 3.0); }
};
template <class S> struct ReadSum { using T = SplitSum<true>; };
template <> struct ReadSum<__half> { using T = SplitSum<false>; };
template <> struct ReadSum<double> { using T = WideSum; };

// FP32 read-out of one instance in box order: thread b takes the box cells
// b, so the four arrays are written once, coalesced, with the zeros off the
// fluid, and the pulls of a row's cells are coalesced too.  80 B are read per fluid
// cell (FP32 storage) and 16 B written per box cell, 87 us for the aorta at the
// copy rate; bound by the sums' arithmetic in FP32 and BF16.  The
// sums must not lose precision against FP64, whose pipe is narrow on this
// part (68 FP64 operations a cell took the whole time before); triples of FP32
// cost about 650 FP32 operations a cell, pairs (FP16) 350.
// Aorta (16.8M box cells, 4.0M fluid): 1,315 us as FP64 gather, four memsets and
// a scatter, in this kernel 238 us (FP16 197); the 96 uneven tubes of a batch
// (33M box cells): 576 launches and 9.3 ms before, 96 launches and 1.42 ms (FP16 1.21).
template <class S>
__global__ void __launch_bounds__(256) k_fields_box(const S *__restrict__ fin, KParams p, const int32_t *__restrict__ rowid,
                                                    int nx, unsigned nbox, float *__restrict__ P, float *__restrict__ jx,
                                                    float *__restrict__ jy, float *__restrict__ jz) {
    using R = typename Storage<S>::R;
    const unsigned b = blockIdx.x * 256u + threadIdx.x;
    if (b >= nbox) return;
    const unsigned line = b / (unsigned)nx;
    const int x = (int)(b - line * (unsigned)nx);
    const int r = __ldg(&rowid[line]);
    float o[4] = {0.f, 0.f, 0.f, 0.f};
    if (r >= 0) {
        const int4 *row = reinterpret_cast<const int4 *>(p.rows + r);
        const int4 h0 = __ldg(row), h1 = __ldg(row + 1), h2 = __ldg(row + 2), h3 = __ldg(row + 3);
        const int k = x - h0.y, c = h0.x + k;
        const uint32_t fl = k >= 0 && k < h0.z ? __ldg(&p.flags[c]) : 0u;
        if (fl & FL_ACTIVE) {
            const int N = (int)p.n;
            const int ln[9] = {h1.z + x, h1.w + x, h2.x + x, h2.y + x, c, h2.w + x, h3.x + x, h3.y + x, h3.z + x};
            R f[NQ];
            f[0] = Storage<S>::ld(fin + c);
#pragma unroll
            for (int i = 1; i < NQ; i++) {
                const int src = ln[nbk(i)] - cx(i), own = c + ((i & 1) ? N : -N);
                f[i] = Storage<S>::ld(fin + (size_t)i * N + (((fl >> i) & 1u) ? own : src));
            }
            typename ReadSum<S>::T s, m[3];
#pragma unroll
            for (int i = 0; i < NQ; i++) {
                s.add(f[i]);
                if (cx(i)) m[0].add(cx(i) > 0 ? f[i] : -f[i]);
                if (cy(i)) m[1].add(cy(i) > 0 ? f[i] : -f[i]);
                if (cz(i)) m[2].add(cz(i) > 0 ? f[i] : -f[i]);
            }
            o[0] = s.pressure();
#pragma unroll
            for (int a = 0; a < 3; a++) o[1 + a] = m[a].value();
            if (!isfinite(s.h)) {  // the plain sum of e_i f_i over all directions (0 times infinity is a NaN)
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    float t = 0.f;
#pragma unroll
                    for (int i = 0; i < NQ; i++)
                        t = __fadd_rn(t, __fmul_rn((float)(a == 0 ? cx(i) : a == 1 ? cy(i) : cz(i)), (float)f[i]));
                    o[1 + a] = t;
                }
            }
        }
    }
    P[b] = o[0];
    jx[b] = o[1];
    jy[b] = o[2];
    jz[b] = o[3];
}

cudaError_t launch_fields_box(int prec, const void *fin, const KParams &p, const int32_t *rowid, int nx, int64_t nbox,
                              float *P, float *jx, float *jy, float *jz, cudaStream_t s) {
    const unsigned grid = (unsigned)((nbox + 255) / 256);
    DISPATCH(prec, (k_fields_box<S><<<grid, 256, 0, s>>>(static_cast<const S *>(fin), p, rowid, nx, (unsigned)nbox, P, jx,
                                                         jy, jz)));
    return cudaGetLastError();
}

cudaError_t launch_wall_shear(int prec, const void *fin, const KParams &p, int c0, int c1, double *out3,
                              cudaStream_t s) {
    const int block = 128;
    const int grid = (c1 - c0 + block - 1) / block;
    if (grid == 0) return cudaSuccess;
    DISPATCH(prec, (k_wall_shear<S><<<grid, block, 0, s>>>(static_cast<const S *>(fin), p, c0, c1, out3)));
    return cudaGetLastError();
}

cudaError_t launch_init_eq(int prec, void *fout, const KParams &p, const double *mac, int c0, int c1,
                           cudaStream_t s) {
    const int block = 256;
    const int grid = (c1 - c0 + block - 1) / block;
    if (grid == 0) return cudaSuccess;
    DISPATCH(prec, (k_init_eq<S><<<grid, block, 0, s>>>(as<S>(fout), p, mac, c0, c1)));
    return cudaGetLastError();
}

cudaError_t launch_cycle_change(const BcKParams &q, const int *bc_first, const int *n_bc, const long long *period,
                                long long steps, double *delta, int n_inst, cudaStream_t s) {
    k_cycle_change<<<n_inst, 256, 0, s>>>(q, bc_first, n_bc, period, steps, delta);
    return cudaGetLastError();
}

cudaError_t launch_init(int prec, void *fout, const KParams &p, const double *f19, int c0, int c1,
                        cudaStream_t s) {
    const int block = 256;
    const int grid = (c1 - c0 + block - 1) / block;
    if (grid == 0) return cudaSuccess;
    DISPATCH(prec, (k_init<S><<<grid, block, 0, s>>>(as<S>(fout), p, f19, c0, c1)));
    return cudaGetLastError();
}

}  // namespace lbm

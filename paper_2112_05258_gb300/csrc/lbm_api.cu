// C-ABI entry points of liblbm (see include/lbm.h for the contract of each).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_internal.h"
#include "lbm_kernels.h"

namespace lbm {
std::string build_layout(const lbm_config *cfg, Layout &L);
}

using namespace lbm;

struct lbm_handle {
    int device = 0;
    int prec = 0;
    int sbytes = 4;  // bytes per stored population
    int rbytes = 4;  // bytes of the compute type
    int block = 256;
    int graph_steps = 64;
    int wave_cap = 8192;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    Layout L;
    std::vector<lbm_instance_desc> inst;  // shapes only (pointers not retained)
    // device buffers
    void *f[2] = {nullptr, nullptr};
    int parity = 0;  // f[parity] holds the resident post-collision state
    void *b = nullptr, *aux = nullptr, *vband = nullptr;
    uint32_t *flags = nullptr;
    RowInfo *rows = nullptr;
    int32_t *chunk_row = nullptr, *rowid = nullptr;
    double *omega = nullptr;
    float *omega_f = nullptr;
    long long *step_dev = nullptr;
    unsigned *status = nullptr;
    BcParam *bc_par = nullptr;
    BcState *bc_state = nullptr;
    int32_t *xf = nullptr, *lk_xb = nullptr, *lk_xf = nullptr, *lk_node = nullptr, *lk_xfi = nullptr;
    uint8_t *lk_i = nullptr;
    double *profile = nullptr, *etab = nullptr, *v0 = nullptr, *wave = nullptr;
    InstParam *inst_dev = nullptr;
    double *partial = nullptr;
    int *arrived = nullptr;
    BcStepResult *bc_result = nullptr;
    int32_t *red_bc = nullptr, *red_chunk = nullptr, *app_bc = nullptr, *app_chunk = nullptr;
    int32_t *band = nullptr, *node_inst = nullptr;
    double *ibX = nullptr, *ibVs = nullptr, *ibI = nullptr, *ibF = nullptr, *ibVf = nullptr;  // FP64 storage
    float *ibD32 = nullptr, *ibVs32 = nullptr, *ibI32 = nullptr, *ibF32 = nullptr, *ibVf32 = nullptr;  // otherwise
    double *ibX0 = nullptr, *ibdA = nullptr, *ibks = nullptr;
    float *ibg0 = nullptr, *ibdA32 = nullptr, *ibks32 = nullptr;
    uint8_t *ibpin = nullptr;
    int32_t *iblines = nullptr, *ibref = nullptr;
    int32_t *fil_nodes = nullptr, *fil_start = nullptr, *fil_count = nullptr;
    double *fil_par = nullptr;
    uint64_t *ibmask = nullptr;
    double *rd_f19 = nullptr, *rd_mac = nullptr;  // read-out scratch, largest instance (allocated on first use)
    // stream-ordered 0D parameter updates: pinned staging ring, one event per slot
    static constexpr int PAR_RING = 64;
    BcParam *par_ring = nullptr, *par_ring_dev = nullptr;  // host and device addresses of the mapped ring
    cudaEvent_t par_ev[PAR_RING] = {};
    int par_pos = 0;
    double *state_rows = nullptr;                  // 8 per boundary, for the asynchronous read
    int64_t max_inst_cells = 0;
    int variant = 0;  // stream-collide occupancy variant (see launch_stream_collide)
    int *inst_bc = nullptr;  // per instance: bc_first, n_bc
    long long *inst_period = nullptr;
    double *inst_delta = nullptr;
    std::vector<void *> allocs;
    int64_t bytes = 0;
    KParams kp{};
    BcKParams bp{};
    IbKParams ibp{};
    int64_t steps = 0;
    // slab pipeline of a step with wall nodes (L.slab_*; n_slab = 0: serial step)
    int n_slab = 0;
    int32_t *node_order = nullptr;
    cudaStream_t s_node = nullptr, s_sc = nullptr;  // wall-node kernels, stream-collide
    std::vector<cudaEvent_t> ev_bm, ev_node, ev_sc;
    cudaEvent_t ev_fork = nullptr;
    // Inside the step graphs, the next step's band velocities run beside this
    // step's 0D boundary kernels: the band entries that are not first-layer
    // cells (band_ind) read no ghost population and no force density that the
    // boundary kernels read, so they start as soon as stream-collide ends (low
    // priority stream s_band); the first-layer band entries (band_dep) follow
    // the boundary kernels (high priority stream s_bc).  Both join the
    // caller's stream before the node kernel.
    bool overlap = false;
    int32_t *band_ind = nullptr, *band_dep = nullptr;
    int n_band_ind = 0, n_band_dep = 0;
    cudaStream_t s_band = nullptr, s_bc = nullptr;
    // Filaments move while stream-collide and the boundary kernels run (step
    // graphs): those read no wall node, and the next node kernel waits for both.
    // The filament kernel is bound by the FP64 pipe, stream-collide by memory:
    // membrane tube of 64 x 64 x 512 with 151 filaments 109.6 -> 95.9 us per step
    // (FP16 99.2 -> 85.7), one of 45 x 45 x 24 30.1 -> 23.9.  Not in FP64, where both are
    // bound by that pipe: 45 x 45 x 24 64.5 -> 79.1, 45 x 45 x 64 106.5 -> 120.9, 64 x 64 x 512
    // 776 -> 760.
    cudaStream_t s_fil = nullptr;
    // A batch's step graphs advance up to four parts of its instances, each a chain
    // of its own (the instances do not meet): while one part's boundary kernels
    // run, bound by latency, the others' stream-collide uses the memory.  A part
    // counts its steps itself.  The boundary kernels have the higher priority:
    // without it they wait until the other parts' stream-collide blocks are all
    // dispatched, and the gain is lost (64 tubes of 14,112 cells in two parts 31.2 us
    // per step, with it 28.8, in one part 30.2).  In 1, 2, 3, 4, 6 parts: those
    // tubes 30.2, 28.7, 26.8, 26.2, 27.6 us per step (FP16 23.0, 22.3, 19.4, 17.7, 18.2;
    // FP64 230, 227, 215, 210, 210), 96 uneven tubes 486, 474, 474, 476, 478 (FP16 370,
    // 357, 356, 356, 358), 8 tubes of 106,920 cells 35.7, 29.0, 27.1, 27.4.
    static constexpr int MAX_PARTS = 4;
    struct Part {
        int c0 = 0, c1 = 0;
        KParams kp{};
        BcKParams bp{};
        cudaStream_t stream = nullptr;  // the first: the lattice's
        cudaEvent_t done = nullptr;
    };
    // (64 tubes of 14,112 cells: building a graph of 100 steps in four parts takes
    // 1.3 ms more than of whole steps, one of 20 less; the rejoining costs 0.3 us a step)
    std::vector<Part> parts;     // empty: one chain
    int part_steps = 0;          // steps of their graph: the first even divisor of graph_steps from 16 on
    cudaEvent_t ev_parts = nullptr;
    long long *step_parts = nullptr;
    cudaEvent_t ev_nodes = nullptr, ev_fil = nullptr;
    cudaEvent_t ev_ofork = nullptr, ev_oband = nullptr, ev_obc = nullptr;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    // for what is left below that: graphs of SHORT_STEPS steps where three or more of
    // them are left, then of one step.  The short ones spare the gaps between single
    // steps and keep what overlaps within a graph: per step of 41 of a 45 x 45 x 24
    // membrane 27.1 -> 24.3 us, of 63 of one of 64 x 64 x 512 103.8 -> 98.1, of 45 of a tube
    // of 500,000 cells 26.8 -> 23.7, of 37 of an aorta of half length 128.1 -> 121.6.  Making
    // one takes about 0.1 ms longer than making the single one, which two do not
    // repay at once (20 steps of a 35 x 35 x 158 membrane on a new lattice 0.70 -> 0.81 ms).
    static constexpr int SHORT_STEPS = 8;
    cudaGraphExec_t graph_short[2] = {nullptr, nullptr}, graph1[2] = {nullptr, nullptr};
    // lbm_step_io: the call's step counter on the device, and its step graphs
    // (each step with its 0D input and output kernels), keyed by the host
    // arrays, the boundary, the graph length and the starting parity
    long long *io_cursor = nullptr;
    struct IoGraph {
        const void *params, *states;
        int np, inst, bc, len, parity;
        cudaGraphExec_t exec;
    };
    std::vector<IoGraph> io_graphs;
    // small lattices: many steps in one launch of so many blocks, clusters or a
    // grid (0: one-step kernels)
    int small_blocks = 0;
    int small_from = 1;  // calls of fewer steps take the one-step kernels all the same
    bool small_on = true;  // lbm_set_multi_step
    size_t small_smem = 0;
    SmallKParams small{};
    // kernel timing
    bool timing = false;
    std::vector<cudaEvent_t> ev;
    size_t ev_used = 0;
    int64_t timed_launches = 0;
    double timed_ms = 0.0;
    std::string err;
};

namespace {

lbm_status fail(lbm_handle *h, lbm_status s, const std::string &msg) {
    if (h) h->err = msg;
    return s;
}

#define CK(h, call)                                                                                 \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess)                                                                      \
            return fail(h, e_ == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA,            \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                       \
    } while (0)

template <class T> cudaError_t dalloc(lbm_handle *h, T **p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, count * sizeof(T));
    if (e != cudaSuccess) return e;
    h->allocs.push_back(q);
    h->bytes += (int64_t)(count * sizeof(T));
    *p = static_cast<T *>(q);
    return cudaSuccess;
}

cudaError_t dalloc_bytes(lbm_handle *h, void **p, size_t bytes) {
    uint8_t *q = nullptr;
    cudaError_t e = dalloc(h, &q, bytes);
    *p = q;
    return e;
}

template <class T> cudaError_t upload(lbm_handle *h, T **p, const std::vector<T> &v) {
    cudaError_t e = dalloc(h, p, v.size());
    if (e != cudaSuccess) return e;
    if (v.empty()) return cudaSuccess;
    return cudaMemcpy(*p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
}

lbm_status check_config(const lbm_config *cfg, std::string &why) {
    if (!cfg) return why = "null config", LBM_ERR_ARG;
    if (cfg->precision < 0 || cfg->precision > 3) return why = "precision out of range", LBM_ERR_ARG;
    if (cfg->n_instances <= 0 || !cfg->inst) return why = "no instances", LBM_ERR_ARG;
    if (cfg->graph_steps < 0 || (cfg->graph_steps % 2) != 0) return why = "graph_steps must be even", LBM_ERR_ARG;
    if (cfg->ib_threads_per_node != 0 && cfg->ib_threads_per_node != 1 && cfg->ib_threads_per_node != 2 &&
        cfg->ib_threads_per_node != 4)
        return why = "ib_threads_per_node must be 0, 1, 2 or 4", LBM_ERR_ARG;
    if (cfg->block_size != 0 && (cfg->block_size < 32 || cfg->block_size > 256 || cfg->block_size % 32))
        return why = "block_size must be a multiple of 32 in [32, 256]", LBM_ERR_ARG;
    for (int q = 0; q < cfg->n_instances; q++) {
        const lbm_instance_desc &d = cfg->inst[q];
        if (d.nx < 1 || d.ny < 1 || d.nz < 1 || !d.node) return why = "bad instance shape or node array", LBM_ERR_ARG;
        if ((double)d.nx * d.ny * d.nz > 2.0e9) return why = "instance too large", LBM_ERR_ARG;
        if (!(d.tau > 0.5)) return why = "tau must exceed 1/2", LBM_ERR_ARG;
        if (d.n_bc < 0 || d.n_bc > MAX_BC || (d.n_bc && !d.bc)) return why = "n_bc out of range", LBM_ERR_ARG;
        const int64_t nbox = (int64_t)d.nx * d.ny * d.nz;
        for (int64_t c = 0; c < nbox; c++)
            if (d.node[c] > 1 + d.n_bc) return why = "node code refers to an undeclared boundary", LBM_ERR_ARG;
        for (int k = 0; k < d.n_bc; k++) {
            const lbm_boundary_desc &b = d.bc[k];
            if (b.kind < 0 || b.kind > 3) return why = "boundary kind out of range", LBM_ERR_ARG;
            if (b.axis < 0 || b.axis > 2 || (b.sign != 1 && b.sign != -1)) return why = "bad boundary normal", LBM_ERR_ARG;
            static const int need[4] = {1, 4, 4, 1};
            if (b.n_params < need[b.kind] || !b.params) return why = "too few boundary params", LBM_ERR_ARG;
            if (b.kind == LBM_BC_RCR && (!(b.params[1] > 0) || !(b.params[2] > 0)))
                return why = "RCR needs C > 0 and R_d > 0", LBM_ERR_ARG;
            if ((b.kind == LBM_BC_RCR || b.kind == LBM_BC_LV) && b.n_params >= 5) {
                const double o = b.params[4];
                if (!(o == 0 || o == 1 || o == 2 || o == 4)) return why = "0D scheme order must be 0, 1, 2 or 4", LBM_ERR_ARG;
            }
            if (b.kind == LBM_BC_LV) {
                if (b.period <= 0 || !b.elastance || (int)b.params[0] != b.period)
                    return why = "LV period and elastance table disagree", LBM_ERR_ARG;
                for (int t = 0; t < b.period; t++)
                    if (!(b.elastance[2 * t] > 0)) return why = "elastance must be positive", LBM_ERR_ARG;
                if (!(b.params[2] > 0)) return why = "N_S must be positive", LBM_ERR_ARG;
            }
        }
        if (d.n_ib < 0 || (d.n_ib > 0 && (!d.ib_X0 || !d.ib_dA || !d.ib_ks || !d.ib_pinned)))
            return why = "bad immersed-boundary arrays", LBM_ERR_ARG;
        if (d.n_ib > 0 && !(d.ib_ms > 0)) return why = "wall mass must be positive", LBM_ERR_ARG;
        for (int64_t s = 0; s < d.n_ib; s++)
            for (int a = 0; a < 3; a++) {
                const int n[3] = {d.nx, d.ny, d.nz};
                const double X = d.ib_X0[3 * s + a];
                if (!(X >= 0.0 && X <= (double)n[a])) return why = "wall node outside the box", LBM_ERR_ARG;
            }
        if (d.ib_n_fil < 0 || (d.ib_n_fil > 0 && (d.n_ib <= 0 || !d.ib_fil_count || !d.ib_fil_nodes || !d.ib_fil_par)))
            return why = "bad filament arrays", LBM_ERR_ARG;
        if (d.ib_n_fil > 0) {
            std::vector<uint8_t> used((size_t)d.n_ib, 0);
            int64_t o = 0;
            for (int64_t k = 0; k < d.ib_n_fil; k++) {
                const int64_t c = d.ib_fil_count[k];
                if (c < 3 || c > LBM_MAX_FILAMENT_NODES) return why = "filament needs 3 to 3072 nodes", LBM_ERR_ARG;
                const double *fp = d.ib_fil_par + 3 * k;
                if (!(fp[0] > 0) || !(fp[1] >= 0) || !(fp[2] >= 0)) return why = "bad filament parameters", LBM_ERR_ARG;
                for (int64_t i = 0; i < c; i++) {
                    const int64_t s = d.ib_fil_nodes[o + i];
                    if (s < 0 || s >= d.n_ib || used[s]) return why = "filament node out of range or repeated", LBM_ERR_ARG;
                    used[s] = 1;
                }
                if (!d.ib_pinned[d.ib_fil_nodes[o]] || !d.ib_pinned[d.ib_fil_nodes[o + c - 1]])
                    return why = "filament end nodes must be pinned", LBM_ERR_ARG;
                o += c;
            }
        }
    }
    return LBM_OK;
}

// One step with the wall-node exchange pipelined over slabs (captured into
// the step graphs only).  Slabs are taken from the highest cells down, so the
// band velocities start on the lines the previous step finished on.  With
// the slab rules of build_slabs:
//   band velocities of slab s        stream A, in slab order
//   node kernel of slab s            stream N, after the band velocities of
//                                    slabs s+1, s, s-1 (the last issued: s-1)
//   stream-collide of slab s         stream C, after the node kernels of
//                                    slabs s+1, s, s-1
//   0D boundary kernels              stream A, after all of them
// The band velocities of slab s clear b there before any node kernel that
// spreads into it (slabs s-1 .. s+1) runs.
lbm_status launch_step_slabs(lbm_handle *h) {
    void *fin = h->f[h->parity], *fout = h->f[1 - h->parity];
    const int K = h->n_slab;
    const Layout &L = h->L;
    CK(h, cudaEventRecord(h->ev_fork, h->stream));
    CK(h, cudaStreamWaitEvent(h->s_node, h->ev_fork, 0));
    CK(h, cudaStreamWaitEvent(h->s_sc, h->ev_fork, 0));
    for (int s = K - 1; s >= 0; s--) {
        CK(h, launch_band_moments(h->prec, fin, h->kp, h->ibp, L.slab_band[s], L.slab_band[s + 1], h->stream));
        CK(h, cudaEventRecord(h->ev_bm[s], h->stream));
    }
    for (int s = K - 1; s >= 0; s--) {
        CK(h, cudaStreamWaitEvent(h->s_node, h->ev_bm[std::max(s - 1, 0)], 0));
        CK(h, launch_ib_nodes(h->prec, h->kp, h->ibp, L.slab_node[s], L.slab_node[s + 1], h->s_node));
        CK(h, cudaEventRecord(h->ev_node[s], h->s_node));
    }
    for (int s = K - 1; s >= 0; s--) {
        CK(h, cudaStreamWaitEvent(h->s_sc, h->ev_node[std::max(s - 1, 0)], 0));
        CK(h, launch_stream_collide(h->prec, fin, fout, h->kp, h->block, h->variant, h->s_sc, 1, L.slab_cell[s],
                                    L.slab_cell[s + 1], s == 0 ? 1 : 0));
        CK(h, cudaEventRecord(h->ev_sc[s], h->s_sc));
    }
    CK(h, cudaStreamWaitEvent(h->stream, h->ev_node[0], 0));
    CK(h, cudaStreamWaitEvent(h->stream, h->ev_sc[0], 0));
    CK(h, launch_boundary(h->prec, fout, h->kp, h->bp, BcIo{}, h->stream));
    h->parity ^= 1;
    return LBM_OK;
}

// One step.  band_done: the band velocities of this step were issued by the
// previous step (next = true there); next: issue the next step's band
// velocities beside this step's boundary kernels (graph capture only; the
// last step of a graph leaves them to the next graph's first step).
lbm_status launch_step(lbm_handle *h, bool timed, bool band_done = false, bool next = false, const BcIo &io = BcIo{}) {
    if (h->n_slab && !timed) return launch_step_slabs(h);
    void *fin = h->f[h->parity], *fout = h->f[1 - h->parity];
    if (h->ibp.n_nodes) CK(h, launch_ib(h->prec, fin, h->kp, h->ibp, h->stream, !band_done));
    const bool fil_aside = h->ibp.n_fil && h->s_fil && h->prec != LBM_F64 && !timed;
    if (fil_aside) {
        CK(h, cudaEventRecord(h->ev_nodes, h->stream));
        CK(h, cudaStreamWaitEvent(h->s_fil, h->ev_nodes, 0));
        CK(h, launch_filaments(h->prec, h->kp, h->ibp, h->s_fil));
        CK(h, cudaEventRecord(h->ev_fil, h->s_fil));
    } else if (h->ibp.n_nodes) {
        CK(h, launch_filaments(h->prec, h->kp, h->ibp, h->stream));
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (timed) {
        if (h->ev_used + 2 > h->ev.size()) {
            // harvest what has been recorded so far
            CK(h, cudaStreamSynchronize(h->stream));
            for (size_t k = 0; k + 1 < h->ev_used; k += 2) {
                float ms = 0.f;
                CK(h, cudaEventElapsedTime(&ms, h->ev[k], h->ev[k + 1]));
                h->timed_ms += ms;
            }
            h->ev_used = 0;
        }
        e0 = h->ev[h->ev_used++];
        e1 = h->ev[h->ev_used++];
        CK(h, cudaEventRecord(e0, h->stream));
    }
    // without wall nodes, every other step runs in descending cell order and
    // starts on the lines the step before finished on (the band-velocity
    // kernel takes that role when there are wall nodes)
    const int desc = h->ibp.n_nodes ? 0 : h->parity;
    CK(h, launch_stream_collide(h->prec, fin, fout, h->kp, h->block, h->variant, h->stream, desc, 0, -1, 1,
                                h->bp.cluster && !timed));
    if (timed) {
        CK(h, cudaEventRecord(e1, h->stream));
        h->timed_launches++;
    }
    if (next && h->overlap && !timed) {
        CK(h, cudaEventRecord(h->ev_ofork, h->stream));
        CK(h, cudaStreamWaitEvent(h->s_band, h->ev_ofork, 0));
        CK(h, cudaStreamWaitEvent(h->s_bc, h->ev_ofork, 0));
        IbKParams ib = h->ibp;
        ib.band = h->band_ind;
        CK(h, launch_band_moments(h->prec, fout, h->kp, ib, 0, h->n_band_ind, h->s_band));
        CK(h, cudaEventRecord(h->ev_oband, h->s_band));
        CK(h, launch_boundary(h->prec, fout, h->kp, h->bp, BcIo{}, h->s_bc));
        ib.band = h->band_dep;
        CK(h, launch_band_moments(h->prec, fout, h->kp, ib, 0, h->n_band_dep, h->s_bc));
        CK(h, cudaEventRecord(h->ev_obc, h->s_bc));
        CK(h, cudaStreamWaitEvent(h->stream, h->ev_oband, 0));
        CK(h, cudaStreamWaitEvent(h->stream, h->ev_obc, 0));
    } else {
        CK(h, launch_boundary(h->prec, fout, h->kp, h->bp, io, h->stream));
    }
    if (fil_aside) CK(h, cudaStreamWaitEvent(h->stream, h->ev_fil, 0));
    h->parity ^= 1;
    return LBM_OK;
}

// len steps of a lattice's parts, each on a stream of its own (captured)
lbm_status launch_parts(lbm_handle *h, int len) {
    CK(h, launch_spread_step(h->step_dev, h->step_parts, (int)h->parts.size(), h->stream));
    CK(h, cudaEventRecord(h->ev_parts, h->stream));
    for (size_t q = 1; q < h->parts.size(); q++) CK(h, cudaStreamWaitEvent(h->parts[q].stream, h->ev_parts, 0));
    for (int k = 0; k < len; k++) {
        for (auto &a : h->parts) {
            cudaStream_t st = a.stream ? a.stream : h->stream;
            void *fin = h->f[h->parity], *fout = h->f[1 - h->parity];
            CK(h, launch_stream_collide(h->prec, fin, fout, a.kp, h->block, h->variant, st, h->parity, a.c0, a.c1, 1,
                                        a.bp.cluster != 0));
            CK(h, launch_boundary(h->prec, fout, a.kp, a.bp, BcIo{}, st));
        }
        h->parity ^= 1;
    }
    for (size_t q = 1; q < h->parts.size(); q++) {
        CK(h, cudaEventRecord(h->parts[q].done, h->parts[q].stream));
        CK(h, cudaStreamWaitEvent(h->stream, h->parts[q].done, 0));
    }
    return LBM_OK;
}

// the graph of len steps from the current parity (captured on first use)
lbm_status ensure_graph(lbm_handle *h, cudaGraphExec_t *graph, int len) {
    const int par = h->parity;
    if (graph[par]) return LBM_OK;
    cudaGraph_t g = nullptr;
    CK(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    lbm_status st = LBM_OK;
    if (!h->parts.empty() && len > 1) st = launch_parts(h, len);
    else
        for (int k = 0; k < len && st == LBM_OK; k++)
            st = launch_step(h, false, k > 0 && h->overlap, k + 1 < len && h->overlap);
    cudaError_t e = cudaStreamEndCapture(h->stream, &g);
    h->parity = par;  // capture does not run anything
    if (st != LBM_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
    }
    CK(h, e);
    e = cudaGraphInstantiateWithFlags(&graph[par], g, cudaGraphInstantiateFlagUseNodePriority);
    cudaGraphDestroy(g);
    CK(h, e);
    return LBM_OK;
}

// One step of lbm_step_io: the params of its row, the step, the state rows
// written after it (rows count from step *io_cursor in the one-launch boundary
// kernel; otherwise *io_cursor counts the call's steps).  band_done / next as in launch_step.
lbm_status launch_io_step(lbm_handle *h, const double *params_dev, int np, int b, double *states_dev, int inst,
                          bool timed, bool band_done, bool next) {
    const InstParam &ip = h->L.inst[inst];
    if (h->bp.cluster)  // the boundary kernel reads and writes the host arrays itself
        return launch_step(h, timed, band_done, next,
                           BcIo{params_dev, states_dev, h->bc_par, h->io_cursor, np, b, ip.bc_first, ip.n_bc});
    CK(h, launch_io_params(params_dev, np, &h->bc_par[b], h->io_cursor, h->stream));
    lbm_status st = launch_step(h, timed, band_done, next);
    if (st != LBM_OK) return st;
    CK(h, launch_io_state(h->bc_state, h->bc_par, h->etab, ip.bc_first, ip.n_bc, (int)h->L.bc.size(), h->step_dev,
                          states_dev, h->io_cursor, h->stream));
    return LBM_OK;
}

// The cached lbm_step_io graph of len steps for these arrays and boundary,
// starting at the current parity (captured on first use).
lbm_status ensure_io_graph(lbm_handle *h, const double *params_dev, int np, int b, double *states_dev, int inst,
                           int len, cudaGraphExec_t *out) {
    for (auto &g : h->io_graphs)
        if (g.params == params_dev && g.states == states_dev && g.np == np && g.inst == inst && g.bc == b &&
            g.len == len && g.parity == h->parity) {
            *out = g.exec;
            return LBM_OK;
        }
    const int par = h->parity;
    cudaGraph_t g = nullptr;
    CK(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    lbm_status st = LBM_OK;
    for (int k = 0; k < len && st == LBM_OK; k++)
        st = launch_io_step(h, params_dev, np, b, states_dev, inst, false, k > 0 && h->overlap,
                            k + 1 < len && h->overlap);
    cudaError_t e = cudaStreamEndCapture(h->stream, &g);
    h->parity = par;  // capture does not run anything
    if (st != LBM_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
    }
    CK(h, e);
    cudaGraphExec_t exec = nullptr;
    e = cudaGraphInstantiateWithFlags(&exec, g, cudaGraphInstantiateFlagUseNodePriority);
    cudaGraphDestroy(g);
    CK(h, e);
    if (h->io_graphs.size() >= 8) {  // a small cache: drop the oldest
        cudaGraphExecDestroy(h->io_graphs.front().exec);
        h->io_graphs.erase(h->io_graphs.begin());
    }
    h->io_graphs.push_back({params_dev, states_dev, np, inst, b, len, par, exec});
    *out = exec;
    return LBM_OK;
}

lbm_status read_gather(lbm_handle *h, int inst, bool with_f) {
    const size_t m = (size_t)h->max_inst_cells;
    if (with_f && !h->rd_f19) CK(h, dalloc(h, &h->rd_f19, 19 * m));
    if (!h->rd_mac) CK(h, dalloc(h, &h->rd_mac, 4 * m));
    const int c0 = (int)h->L.inst_cell_begin[inst], c1 = (int)h->L.inst_cell_end[inst];
    CK(h, launch_gather(h->prec, h->f[h->parity], h->kp, c0, c1, with_f ? h->rd_f19 : nullptr, h->rd_mac,
                        h->stream));
    return LBM_OK;
}

void drop_graphs(lbm_handle *h) {
    for (auto &g : h->io_graphs) cudaGraphExecDestroy(g.exec);
    h->io_graphs.clear();
    for (int k = 0; k < 2; k++) {
        if (h->graph[k]) {
            cudaGraphExecDestroy(h->graph[k]);
            h->graph[k] = nullptr;
        }
        if (h->graph_short[k]) {
            cudaGraphExecDestroy(h->graph_short[k]);
            h->graph_short[k] = nullptr;
        }
        if (h->graph1[k]) {
            cudaGraphExecDestroy(h->graph1[k]);
            h->graph1[k] = nullptr;
        }
    }
}

// Decides whether the lattice takes its steps in the multi-step kernel, and
// with how many blocks per instance.
cudaError_t set_up_small(lbm_handle *h) {
    const Layout &L = h->L;
    if (!L.ib_dA.empty() || L.n_fluid == 0) return cudaSuccess;
    if (L.n_fluid > 160 * 2700) return cudaSuccess;  // beyond the shared memory of all blocks
    std::vector<int32_t> bulk, off;
    int64_t worst_bulk[17] = {0};
    size_t smem_b = 0;
    int most_bc = 0, worst_xf = 0;
    std::vector<uint8_t> seen((size_t)L.n_stored, 0);
    for (size_t q = 0; q < L.inst.size(); q++) {
        const InstParam &ip = L.inst[q];
        most_bc = std::max(most_bc, ip.n_bc);
        for (int k = 0; k < ip.n_bc; k++) {
            const BcParam &b = L.bc[ip.bc_first + k];
            if (b.n_red > SMALL_MAX_RED || b.n_nodes > 32767) return cudaSuccess;
            worst_xf = std::max(worst_xf, b.n_xf);
            smem_b = std::max(smem_b, small_smem_boundary(b.n_xf, b.n_links, b.n_nodes, h->prec == LBM_F64));
            for (int a = 0; a < b.n_xf; a++) {
                uint8_t &c = seen[(size_t)L.xf[b.xf_off + a]];
                if (c) return cudaSuccess;  // a cell in two first layers
                c = 1;
            }
        }
        off.push_back((int32_t)bulk.size());
        for (int64_t c = L.inst_cell_begin[q]; c < L.inst_cell_end[q]; c++)
            if ((L.flags[(size_t)c] & FL_ACTIVE) && !seen[(size_t)c]) bulk.push_back((int32_t)c);
        const int64_t n = (int64_t)bulk.size() - off.back();
        for (int C = ip.n_bc + 1; C <= 16; C++)
            worst_bulk[C] = std::max(worst_bulk[C], (n + C - ip.n_bc - 1) / (C - ip.n_bc));
    }
    off.push_back((int32_t)bulk.size());
    // Times of a step in us, measured on GB300 over tubes of 900 to 320,000
    // cells.  This kernel: as many rounds as the clusters need, each the longer
    // of the boundary block (latency: 3.1 us and its first layer's share; FP64
    // runs on a pipe of 2 lanes an SM) and of a bulk block's cells.  One-step
    // kernels: launches and latencies of 12 us (FP64: 21), then bandwidth.
    const bool f64 = h->prec == LBM_F64;
    const double cells = (double)L.n_fluid;
    // Without boundaries a one-step kernel is all there is to a step.  FP32 calls of 100 steps
    // of closed boxes, one-step kernels -> this one: 55,000 cells 308 -> 322 us, 135,000 410 ->
    // 455 (406 and 516 before the short graphs), 217,000 551 -> 649, 340,000 712 -> 828; of 24
    // steps 74 -> 82, 100 -> 114, 135 -> 161, 172 -> 205.
    if (!f64 && L.bc.empty() && cells > 170e3) return cudaSuccess;
    const double one_step = std::max(f64 ? 21.0 : 12.0, (f64 ? 16.0 : 9.0) + cells * (f64 ? 240e-6 : 30e-6));
    double best = 0.9 * one_step, t_small = 0.0;
    for (int C : {16, 8}) {
        if (C <= most_bc) continue;
        const size_t smem = std::max(smem_b, small_smem_bulk((int)worst_bulk[C]));
        if (smem > SMALL_MAX_SMEM) continue;
        const double owner = f64 ? 3.5 + 0.085 * worst_xf : 3.1 + 0.0058 * worst_xf;
        const double bulk = f64 ? 1.5 + 33e-3 * worst_bulk[C] : 0.7 + 3.2e-3 * worst_bulk[C];
        if (std::max(owner, bulk) >= best) continue;
        int clusters = 0;
        if (prepare_small(h->prec, C, smem, &clusters) != cudaSuccess || clusters < 1) {
            (void)cudaGetLastError();
            continue;
        }
        const int rounds = ((int)L.inst.size() + clusters - 1) / clusters;
        const double t = rounds * std::max(owner, bulk);
        if (t >= best) continue;
        best = t_small = t;
        h->small.cluster = C;
        h->small_blocks = C * (int)L.inst.size();
        h->small_smem = smem;
    }
    // One grid over all instances, if that beats the better of the two (by 5 %, as
    // it takes more SMs): a boundary block as above (FP32: another pass beyond 768
    // cells), and as many bulk blocks as are done a little earlier, if the shared
    // memory of those takes their cells; the other SMs stay free for other streams.
    // (Lattices stepped at once on streams of their own take turns; a caller can choose
    // the one-step kernels for them, lbm_set_multi_step, where the figures stand.  One
    // alone 7.2 instead of 12.4 us a step, beside a stream of long kernels 16 instead of 328.)
    int sms = 0, per_sm = 0;
    const int nb = (int)L.bc.size();
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
    if (e == cudaSuccess && nb < sms) {
        const double owner = f64 ? std::max(6.6 + 0.048 * worst_xf, 1.7 + 0.084 * worst_xf)
                                 : 3.1 + 0.0071 * worst_xf + 1.4 * (std::max(worst_xf - 1, 0) / 768);
        const double b0 = f64 ? 1.5 : 2.05, b1 = f64 ? 34.5e-3 : 2.63e-3, n = (double)bulk.size();
        const double fit = std::min((0.9 * owner - b0) / b1, f64 ? 2500.0 : 2600.0);
        const int w = (int)std::max(1.0, std::min((double)(sms - nb), std::ceil(n / fit)));
        const double per = std::ceil(n / w), t = std::max(owner, b0 + b1 * per);
        const size_t smem = std::max(smem_b, small_smem_grid((int)per, f64));
        if (t < 0.95 * (h->small_blocks ? best : one_step) && smem <= SMALL_MAX_SMEM) {
            if (prepare_small(h->prec, 0, smem, &per_sm) == cudaSuccess && per_sm >= 1) {
                t_small = t;
                h->small.cluster = 0;
                h->small_blocks = nb + w;
                h->small_smem = smem;
            }
            (void)cudaGetLastError();
        }
    }
    if (e != cudaSuccess || !h->small_blocks) return e;
    // A launch lays out its tables first (8.4 us), which a call of one step does not repay where
    // the step is long: such calls take the one-step kernels.  us for a call of one step, queued
    // and waited for, one-step kernels -> this one: FP32 2,400 cells 11.4, 26.3 -> 11.2, 27.4, 24x24x64
    // tube 12.4, 26.2 -> 12.4, 28.2, 50,283 cells 12.4, 27.4 -> 14.4, 30.1, 324,139 cells 17.9, 32.1 ->
    // 20.6, 36.9, 10,330 cells behind 1,029 first-layer ones 16.5, 30.0 -> 22.6, 38.7, 16 tubes of
    // 14,112 cells 14.7, 30.9 -> 14.4, 30.7; FP64 2,400 cells 22.6, 36.7 -> 18.4, 34.8, 24x24x64 tube 22.6,
    // 37.4 -> 26.7, 42.6, 176,407 cells 63.6, 77.5 -> 56.0, 74.6.  Two steps repay it, without boundaries
    // (6.2 -> 8.3 to 10.3) three in FP32.
    const double single = f64 ? 21.5 + 235e-6 * cells : 11.4 + 0.1 * ((double)L.inst.size() - 1) + 20e-6 * cells;
    h->small_from = L.bc.empty() ? (f64 ? 2 : 3) : 8.4 + t_small > single ? 2 : 1;
    int32_t *d_bulk = nullptr, *d_off = nullptr;
    int *done = nullptr;
    unsigned *meet = nullptr;
    if (e == cudaSuccess) e = upload(h, &d_bulk, bulk);
    if (e == cudaSuccess) e = dalloc(h, &meet, 1);
    if (e == cudaSuccess) e = cudaMemset(meet, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = upload(h, &d_off, off);
    if (e == cudaSuccess) e = dalloc(h, &done, 1);
    if (e == cudaSuccess) e = cudaMemset(done, 0, sizeof(int));
    h->small.inst = h->inst_dev;
    h->small.bulk = d_bulk;
    h->small.bulk_off = d_off;
    h->small.done = done;
    h->small.meet = meet;
    h->small.polls = SMALL_POLLS;
    h->small.n_inst = (int)L.inst.size();
    h->small.par = h->bc_par;
    return e;
}

// n steps in the multi-step kernel (launches of at most SMALL_MAX_STEPS
// steps); io: per-step params and state rows of lbm_step_io, or null.
lbm_status small_steps(lbm_handle *h, int64_t n, const SmallKParams *io = nullptr) {
    if (n == 0) return LBM_OK;
    SmallKParams sp = io ? *io : h->small;
    // refused as the step graphs of the other lattices are: a replay would pass the host's step count by
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    CK(h, cudaStreamIsCapturing(h->stream, &capture));
    if (capture != cudaStreamCaptureStatusNone) return fail(h, LBM_ERR_CUDA, "the stream is being captured");
    while (n > 0) {
        sp.n_steps = (int)std::min<int64_t>(n, SMALL_MAX_STEPS);
        CK(h, launch_small(h->prec, h->f[h->parity], h->f[1 - h->parity], h->kp, h->bp, sp, h->small_blocks,
                           h->small_smem, h->stream));
        if (sp.n_steps & 1) h->parity ^= 1;
        h->steps += sp.n_steps;
        n -= sp.n_steps;
        if (sp.io_params) sp.io_params += (size_t)sp.n_steps * sp.io_np;
        if (sp.io_states) sp.io_states += (size_t)sp.n_steps * 8 * sp.io_nb;
    }
    return LBM_OK;
}

// Candidates of lbm_autotune without wall nodes are timed as the step graphs run
// them: stream-collide and the boundary kernels of every part, each part on its
// stream.  Timed by stream-collide alone over all cells, the shape picked for 64
// tubes of 14,112 cells (FP32) took 30.6 us per step where the default takes 26.8.
// The steps all begin from the resident populations and write the other buffer,
// which the next real step overwrites; the 0D state, closure velocities, waveforms
// and step counters are scratch copies.
struct TuneScratch {
    std::vector<void *> mem;
    std::vector<lbm_handle::Part> parts;
    ~TuneScratch() {
        for (void *p : mem) cudaFree(p);
    }
    cudaError_t get(void **p, size_t bytes) {
        const cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 8));
        if (e == cudaSuccess) mem.push_back(*p);
        return e;
    }
};
lbm_status tune_scratch(lbm_handle *h, TuneScratch &t) {
    const size_t nb = std::max<size_t>(1, h->L.bc.size()), nxf = std::max<size_t>(1, h->L.xf.size());
    t.parts = h->parts;
    if (t.parts.empty()) {  // the whole lattice
        t.parts.emplace_back();
        t.parts[0].c1 = h->kp.cells;
        t.parts[0].kp = h->kp;
        t.parts[0].bp = h->bp;
    }
    void *state = nullptr, *v0 = nullptr, *wave = nullptr, *step = nullptr;
    CK(h, t.get(&state, 2 * nb * sizeof(BcState)));
    CK(h, t.get(&v0, 3 * nxf * sizeof(double)));
    CK(h, t.get(&wave, nb * 4 * sizeof(double)));
    CK(h, t.get(&step, t.parts.size() * sizeof(long long)));
    CK(h, cudaMemcpyAsync(state, h->bc_state, 2 * nb * sizeof(BcState), cudaMemcpyDeviceToDevice, h->stream));
    CK(h, cudaMemcpyAsync(v0, h->v0, 3 * nxf * sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
    CK(h, launch_spread_step(h->step_dev, static_cast<long long *>(step), (int)t.parts.size(), h->stream));
    for (size_t q = 0; q < t.parts.size(); q++) {
        lbm_handle::Part &a = t.parts[q];
        a.kp.step = static_cast<long long *>(step) + q;
        a.bp.state = static_cast<BcState *>(state);
        a.bp.v0 = static_cast<double *>(v0);
        a.bp.wave = static_cast<double *>(wave);
        a.bp.wave_cap = 1;
    }
    return LBM_OK;
}
lbm_status tune_steps(lbm_handle *h, const TuneScratch &t, int block, int variant, int len) {
    void *fin = h->f[h->parity], *fout = h->f[1 - h->parity];
    if (t.parts.size() > 1) CK(h, cudaEventRecord(h->ev_parts, h->stream));
    for (size_t q = 1; q < t.parts.size(); q++) CK(h, cudaStreamWaitEvent(t.parts[q].stream, h->ev_parts, 0));
    for (int k = 0; k < len; k++)
        for (auto &a : t.parts) {
            cudaStream_t st = a.stream ? a.stream : h->stream;
            CK(h, launch_stream_collide(h->prec, fin, fout, a.kp, block, variant, st, k & 1, a.c0, a.c1, 1,
                                        a.bp.cluster != 0));
            CK(h, launch_boundary(h->prec, fout, a.kp, a.bp, BcIo{}, st));
        }
    for (size_t q = 1; q < t.parts.size(); q++) {
        CK(h, cudaEventRecord(t.parts[q].done, t.parts[q].stream));
        CK(h, cudaStreamWaitEvent(h->stream, t.parts[q].done, 0));
    }
    return LBM_OK;
}
// mean time of a step of len * reps, after one graph of warm-up
lbm_status tune_candidate(lbm_handle *h, const TuneScratch &t, int block, int variant, int len, int reps,
                          cudaEvent_t e0, cudaEvent_t e1, float *ms) {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
    CK(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    const lbm_status st = tune_steps(h, t, block, variant, len);
    cudaError_t e = cudaStreamEndCapture(h->stream, &g);
    if (st == LBM_OK && e == cudaSuccess) e = cudaGraphInstantiateWithFlags(&x, g, cudaGraphInstantiateFlagUseNodePriority);
    if (g) cudaGraphDestroy(g);
    if (st != LBM_OK) return st;
    if (e == cudaSuccess) e = cudaGraphLaunch(x, h->stream);
    if (e == cudaSuccess) e = cudaEventRecord(e0, h->stream);
    for (int k = 0; k < reps && e == cudaSuccess; k++) e = cudaGraphLaunch(x, h->stream);
    if (e == cudaSuccess) e = cudaEventRecord(e1, h->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
    if (x) cudaGraphExecDestroy(x);
    CK(h, e);
    *ms /= (float)(len * reps);
    return LBM_OK;
}

bool bad_inst(lbm_handle *h, int inst) { return !h || inst < 0 || inst >= (int)h->inst.size(); }

// validation of one set of boundary params (lbm_set_0d_params, lbm_step_io); null if valid
const char *bad_params(const BcParam &bp, const double *p, int np) {
    static const int need[4] = {1, 4, 4, 1};
    if (np < need[bp.kind]) return "too few params";
    if (bp.kind == BC_RCR && (!(p[1] > 0) || !(p[2] > 0))) return "RCR needs C, R_d > 0";
    if (bp.kind == BC_LV && ((int)p[0] != bp.period || !(p[2] > 0))) return "LV period is fixed at creation; N_S > 0";
    if ((bp.kind == BC_RCR || bp.kind == BC_LV) && np >= 5 && !(p[4] == 0 || p[4] == 1 || p[4] == 2 || p[4] == 4))
        return "0D scheme order must be 0, 1, 2 or 4";
    return nullptr;
}

}  // namespace

extern "C" {

lbm_status lbm_check_config(const lbm_config *cfg, lbm_layout_stats *stats, char *why, int why_len) {
    std::string msg;
    lbm_status st = check_config(cfg, msg);
    Layout L;
    if (st == LBM_OK) {
        msg = build_layout(cfg, L);
        if (msg.empty() && (double)NQ * (double)population_cells(L.n_stored) >= 2147483647.0)
            msg = "more than 2^31 / 19 stored cells (32-bit population offsets)";
        st = msg.empty() ? LBM_OK : LBM_ERR_ARG;
    }
    if (why && why_len > 0) {
        const size_t n = std::min(msg.size(), (size_t)why_len - 1);
        memcpy(why, msg.data(), n);
        why[n] = 0;
    }
    if (st == LBM_OK && stats) {
        stats->fluid_cells = L.n_fluid;
        stats->stored_cells = L.n_stored;
        stats->box_cells = L.n_box;
        stats->band_cells = (int64_t)L.band.size();
        stats->links = (int64_t)L.lk_xb.size();
        stats->ib_nodes = (int64_t)L.ib_dA.size();
        stats->filaments = (int64_t)L.fil_start.size();
        stats->slabs = 0;
        if (cfg->ib_slabs > 1) {
            build_slabs(L, cfg->ib_slabs);
            if (!L.slab_cell.empty()) stats->slabs = (int64_t)L.slab_cell.size() - 1;
        }
    }
    return st;
}

lbm_status lbm_create(const lbm_config *cfg, lbm_handle **out) {
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    std::string why;
    if (check_config(cfg, why) != LBM_OK) {
        fprintf(stderr, "lbm_create: %s\n", why.c_str());
        return LBM_ERR_ARG;
    }
    lbm_handle *h = new lbm_handle();
    h->device = cfg->device;
    h->prec = cfg->precision;
    static const int sb[4] = {4, 2, 2, 8};
    h->sbytes = sb[h->prec];
    h->rbytes = h->prec == LBM_F64 ? 8 : 4;
    h->block = cfg->block_size ? cfg->block_size : 128;
    h->graph_steps = cfg->graph_steps ? cfg->graph_steps : 64;
    h->wave_cap = cfg->wave_capacity > 0 ? cfg->wave_capacity : 8192;
    h->inst.assign(cfg->inst, cfg->inst + cfg->n_instances);
    for (auto &d : h->inst) {
        d.node = nullptr;
        d.bc = nullptr;
        d.ib_X0 = d.ib_dA = d.ib_ks = nullptr;
        d.ib_pinned = nullptr;
        d.ib_fil_count = d.ib_fil_nodes = nullptr;
        d.ib_fil_par = nullptr;
    }
    auto bail = [&](lbm_status s, const std::string &m) {
        fprintf(stderr, "lbm_create: %s\n", m.c_str());
        lbm_destroy(h);
        return s;
    };
    std::string e = build_layout(cfg, h->L);
    if (!e.empty()) return bail(LBM_ERR_ARG, e);
    Layout &L = h->L;
    if ((double)NQ * (double)population_cells(L.n_stored) >= 2147483647.0)
        return bail(LBM_ERR_ARG, "more than 2^31 / 19 stored cells (32-bit population offsets)");
    if (cudaSetDevice(h->device) != cudaSuccess) return bail(LBM_ERR_CUDA, "cudaSetDevice failed");
    if (cfg->stream) {
        h->stream = static_cast<cudaStream_t>(cfg->stream);
    } else {
        if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess)
            return bail(LBM_ERR_CUDA, "stream creation failed");
        h->own_stream = true;
    }
    const size_t n = (size_t)L.n_stored;
    auto ck = [&](cudaError_t ce, const char *what) -> bool {
        if (ce == cudaSuccess) return true;
        h->err = std::string(what) + ": " + cudaGetErrorString(ce);
        return false;
    };
    bool ok = true;
    for (int k = 0; k < 2 && ok; k++) {
        const size_t pop_bytes = (size_t)NQ * (size_t)population_cells((int64_t)n) * h->sbytes;
        ok = ck(dalloc_bytes(h, &h->f[k], pop_bytes), "populations");
        if (ok) ok = ck(cudaMemset(h->f[k], 0, pop_bytes), "memset");
    }
    if (ok) ok = ck(dalloc_bytes(h, &h->b, 4 * n * h->rbytes), "b") && ck(cudaMemset(h->b, 0, 4 * n * h->rbytes), "memset");
    if (ok) ok = ck(dalloc_bytes(h, &h->aux, 4 * (size_t)population_cells((int64_t)n) * h->rbytes), "aux") &&
                 ck(cudaMemset(h->aux, 0, 4 * (size_t)population_cells((int64_t)n) * h->rbytes), "memset");
    if (ok) ok = ck(upload(h, &h->flags, L.flags), "flags");
    if (ok) ok = ck(upload(h, &h->rows, L.rows), "rows");
    if (ok) ok = ck(upload(h, &h->chunk_row, L.chunk_row), "chunks");
    if (ok) ok = ck(upload(h, &h->rowid, L.rowid), "rowid");
    std::vector<double> om;
    for (auto &ip : L.inst) om.push_back(ip.omega);
    std::vector<float> omf(om.begin(), om.end());
    if (ok) ok = ck(upload(h, &h->omega, om), "omega") && ck(upload(h, &h->omega_f, omf), "omega");
    if (ok) ok = ck(upload(h, &h->inst_dev, L.inst), "instances");
    long long minus1 = -1;
    if (ok) ok = ck(dalloc(h, &h->step_dev, 1), "step") &&
                 ck(cudaMemcpy(h->step_dev, &minus1, sizeof minus1, cudaMemcpyHostToDevice), "step");
    if (ok) ok = ck(dalloc(h, &h->status, 1), "status") && ck(cudaMemset(h->status, 0, sizeof(unsigned)), "status");
    // 0D boundaries
    std::vector<BcState> st(L.bc.size());
    for (size_t k = 0; k < L.bc.size(); k++) {
        memset(&st[k], 0, sizeof(BcState));
        if (L.bc[k].kind == BC_RCR) st[k].Pw = L.bc[k].par[3];
        if (L.bc[k].kind == BC_LV) {
            st[k].Pv = L.bc[k].par[3];
            st[k].Td = -1e300;
        }
    }
    std::vector<BcState> st2(st);
    st2.insert(st2.end(), st.begin(), st.end());  // [2][n_bc]: read n & 1, write (n + 1) & 1
    if (ok) ok = ck(upload(h, &h->bc_par, L.bc), "bc") && ck(upload(h, &h->bc_state, st2), "bc state");
    if (ok) ok = ck(dalloc(h, &h->arrived, std::max<size_t>(1, L.bc.size())), "arrivals") &&
                 ck(cudaMemset(h->arrived, 0, std::max<size_t>(1, L.bc.size()) * sizeof(int)), "arrivals") &&
                 ck(dalloc(h, &h->bc_result, std::max<size_t>(1, L.bc.size())), "step results");
    if (ok) ok = ck(dalloc(h, &h->partial, 2 * std::max<size_t>(1, (size_t)L.n_partial)), "partials") &&
                 ck(upload(h, &h->red_bc, L.red_bc), "tables") && ck(upload(h, &h->red_chunk, L.red_chunk), "tables") &&
                 ck(upload(h, &h->app_bc, L.app_bc), "tables") && ck(upload(h, &h->app_chunk, L.app_chunk), "tables");
    if (ok) ok = ck(upload(h, &h->xf, L.xf), "xf") && ck(upload(h, &h->lk_xb, L.lk_xb), "links") &&
                 ck(upload(h, &h->lk_xf, L.lk_xf), "links") && ck(upload(h, &h->lk_node, L.lk_node), "links") &&
                 ck(upload(h, &h->lk_xfi, L.lk_xfi), "links") && ck(upload(h, &h->lk_i, L.lk_i), "links") &&
                 ck(upload(h, &h->profile, L.profile), "profile") && ck(upload(h, &h->etab, L.etab), "etab");
    if (ok) ok = ck(dalloc(h, &h->v0, 3 * std::max<size_t>(1, L.xf.size())), "v0") &&
                 ck(cudaMemset(h->v0, 0, 3 * std::max<size_t>(1, L.xf.size()) * sizeof(double)), "v0");
    const size_t nwave = (size_t)h->wave_cap * std::max<size_t>(1, L.bc.size()) * 4;
    if (ok) ok = ck(dalloc(h, &h->wave, nwave), "wave") && ck(cudaMemset(h->wave, 0, nwave * sizeof(double)), "wave");
    // immersed boundary
    const size_t ns = L.ib_dA.size();
    if (ok && ns) {
        std::vector<int32_t> ni;
        for (size_t q = 0; q < L.inst.size(); q++)
            for (int s = 0; s < L.inst[q].n_ib; s++) ni.push_back((int32_t)q);
        std::vector<double> zero(3 * ns, 0.0);
        std::vector<float> zero32(3 * ns, 0.0f);
        std::vector<float> dA32(L.ib_dA.begin(), L.ib_dA.end()), ks32(L.ib_ks.begin(), L.ib_ks.end());
        // the node state in the arithmetic's precision (FP32: displacements from X0)
        const bool st64 = h->prec == LBM_F64;
        ok = ck(upload(h, &h->band, L.band), "band") && ck(upload(h, &h->node_inst, ni), "ib") &&
             (st64 ? ck(upload(h, &h->ibX, L.ib_X0), "ib") && ck(upload(h, &h->ibVs, zero), "ib") &&
                         ck(upload(h, &h->ibI, zero), "ib") && ck(upload(h, &h->ibF, zero), "ib") &&
                         ck(upload(h, &h->ibVf, zero), "ib")
                   : ck(upload(h, &h->ibD32, zero32), "ib") && ck(upload(h, &h->ibVs32, zero32), "ib") &&
                         ck(upload(h, &h->ibI32, zero32), "ib") && ck(upload(h, &h->ibF32, zero32), "ib") &&
                         ck(upload(h, &h->ibVf32, zero32), "ib") && ck(upload(h, &h->ibg0, L.ib_g0), "ib") &&
                         ck(upload(h, &h->ibdA32, dA32), "ib") && ck(upload(h, &h->ibks32, ks32), "ib")) &&
             ck(upload(h, &h->ibX0, L.ib_X0), "ib") &&
             ck(upload(h, &h->ibdA, L.ib_dA), "ib") && ck(upload(h, &h->ibks, L.ib_ks), "ib") &&
             ck(upload(h, &h->ibpin, L.ib_pinned), "ib") && ck(upload(h, &h->iblines, L.ib_lines), "ib") &&
             ck(upload(h, &h->ibmask, L.ib_mask), "ib") && ck(upload(h, &h->ibref, L.ib_ref), "ib") &&
             ck(upload(h, &h->fil_nodes, L.fil_nodes), "filaments") &&
             ck(upload(h, &h->fil_start, L.fil_start), "filaments") &&
             ck(upload(h, &h->fil_count, L.fil_count), "filaments") &&
             ck(upload(h, &h->fil_par, L.fil_par), "filaments") &&
             (L.fil_start.empty() || ck(prepare_filament_kernel(L.max_fil), "filament kernel")) &&
             ck(dalloc_bytes(h, &h->vband, 4 * n * h->rbytes), "vband") &&
             ck(cudaMemset(h->vband, 0, 4 * n * h->rbytes), "vband");
    }
    {
        std::vector<int> ib2;  // bc_first of every instance, then n_bc of every instance
        for (auto &ip : L.inst) ib2.push_back(ip.bc_first);
        for (auto &ip : L.inst) ib2.push_back(ip.n_bc);
        for (size_t q = 0; q < L.inst.size(); q++)
            h->max_inst_cells = std::max<int64_t>(h->max_inst_cells, L.inst_cell_end[q] - L.inst_cell_begin[q]);
        if (ok) ok = ck(upload(h, &h->inst_bc, ib2), "instances") &&
                     ck(dalloc(h, &h->inst_period, L.inst.size()), "instances") &&
                     ck(dalloc(h, &h->inst_delta, L.inst.size()), "instances");
    }
    if (!ok) {
        lbm_status s = h->err.find("out of memory") != std::string::npos ? LBM_ERR_OOM : LBM_ERR_CUDA;
        return bail(s, h->err);
    }
    h->kp.n = (long long)population_cells((int64_t)n);
    h->kp.cells = (int)n;
    h->kp.flags = h->flags;
    h->kp.rows = h->rows;
    h->kp.chunk_row = h->chunk_row;
    h->kp.omega = h->omega;
    h->kp.omega_f = h->omega_f;
    h->kp.b = h->b;
    h->kp.aux = h->aux;
    h->kp.step = h->step_dev;
    h->kp.status = h->status;
    // Prefetch and kept stores of stream-collide (its LARGE kernels): where the two buffers of
    // populations exceed the L2; in FP64, which is bound by its pipe, and with wall nodes, whose
    // kernels want the L2 too, where one does.  us per step without -> with (one buffer of so many
    // MB): batches FP32 33 MB 15.56 -> 15.73, 67 28.6 -> 27.0, 70 27.1 -> 26.2, 106 42.8 -> 42.0; FP16
    // 35 MB 19.0 -> 21.5, 53 32.6 -> 33.8, 74 39.5 -> 38.6, 90 52.0 -> 48.1, 107 68.4 -> 62.2; single tubes
    // FP32 49 MB 26.2 -> 26.9, 79 37.4 -> 37.3, FP16 39 MB 28.7 -> 29.2, 97 58.0 -> 56.7.
    const size_t pop_bytes = (size_t)NQ * n * h->sbytes;
    const bool one_exceeds = exceeds_l2(pop_bytes, h->device);
    h->kp.keep = h->prec == LBM_F64 || ns ? one_exceeds : exceeds_l2(2 * pop_bytes, h->device);
    h->bp.n_bc_total = h->bp.n_bc = (int)L.bc.size();
    h->bp.par = h->bc_par;
    h->bp.state = h->bc_state;
    h->bp.xf = h->xf;
    h->bp.lk_xb = h->lk_xb;
    h->bp.lk_xf = h->lk_xf;
    h->bp.lk_node = h->lk_node;
    h->bp.lk_xfi = h->lk_xfi;
    h->bp.lk_i = h->lk_i;
    h->bp.profile = h->profile;
    h->bp.etab = h->etab;
    h->bp.v0 = h->v0;
    h->bp.wave = h->wave;
    h->bp.wave_cap = h->wave_cap;
    h->bp.partial = h->partial;
    h->bp.arrived = h->arrived;
    {
        // the per-block 0D step costs nothing extra while the link blocks run
        // in one wave (about 4 resident per SM); beyond that, once per boundary
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess) sms = 1;
        h->bp.step_in_reduce = (int)L.app_bc.size() > 4 * sms ? 1 : 0;
    }
    h->bp.result = h->bc_result;
    h->bp.cluster = h->bp.wide = 0;
    if (L.ib_dA.empty()) {
        // one launch for the boundary work: blocks enough that a thread has one
        // link (at most 8 blocks of 512 per boundary), as long as all clusters
        // run at once; the figures for the line stand at k_boundary
        int links = 0;
        for (auto &b : L.bc) links = std::max(links, b.n_links);
        h->bp.wide = links > 4 * 256;
        int c = 1;
        while (c < 8 && c * (h->bp.wide ? 512 : 256) < links) c *= 2;
        const int most = h->bp.wide ? 200 : 300;  // blocks of 512 threads: one per SM
        if (h->prec != LBM_F64 && links > 0 && links <= 4096 && c * (int)L.bc.size() <= most) h->bp.cluster = c;
    }
    h->bp.n_red_blocks = (int)L.red_bc.size();
    h->bp.n_app_blocks = (int)L.app_bc.size();
    h->bp.red_bc = h->red_bc;
    h->bp.red_chunk = h->red_chunk;
    h->bp.app_bc = h->app_bc;
    h->bp.app_chunk = h->app_chunk;
    h->ibp.n_nodes = (int)ns;
    h->ibp.n_band = (int)L.band.size();
    h->ibp.band = h->band;
    h->ibp.node_inst = h->node_inst;
    h->ibp.inst = h->inst_dev;
    h->ibp.rowid = h->rowid;
    h->ibp.X = h->ibX;
    h->ibp.Vs = h->ibVs;
    h->ibp.I = h->ibI;
    h->ibp.F = h->ibF;
    h->ibp.Vf = h->ibVf;
    h->ibp.D32 = h->ibD32;
    h->ibp.Vs32 = h->ibVs32;
    h->ibp.I32 = h->ibI32;
    h->ibp.F32 = h->ibF32;
    h->ibp.Vf32 = h->ibVf32;
    h->ibp.g0 = h->ibg0;
    h->ibp.dA32 = h->ibdA32;
    h->ibp.ks32 = h->ibks32;
    h->ibp.X0 = h->ibX0;
    h->ibp.dA = h->ibdA;
    h->ibp.ks = h->ibks;
    h->ibp.pinned = h->ibpin;
    h->ibp.vband = h->vband;
    h->ibp.threads_per_node = cfg->ib_threads_per_node ? cfg->ib_threads_per_node : 4;
    h->ibp.lines = h->iblines;
    h->ibp.mask = h->ibmask;
    h->ibp.ref = h->ibref;
    h->ibp.n_fil = (int)L.fil_start.size();
    h->ibp.max_fil = L.max_fil;
    h->ibp.fil_nodes = h->fil_nodes;
    h->ibp.fil_start = h->fil_start;
    h->ibp.fil_count = h->fil_count;
    h->ibp.fil_par = h->fil_par;
    h->ibp.order = nullptr;
    if (ns && cfg->ib_slabs > 1) {
        build_slabs(L, cfg->ib_slabs);
        if (!L.slab_cell.empty()) {
            const int K = (int)L.slab_cell.size() - 1;
            int lo = 0, hi = 0;
            bool sok = ck(upload(h, &h->node_order, L.node_order), "node order") &&
                       ck(cudaDeviceGetStreamPriorityRange(&lo, &hi), "stream priorities") &&
                       ck(cudaStreamCreateWithPriority(&h->s_node, cudaStreamNonBlocking, hi), "streams") &&
                       ck(cudaStreamCreateWithPriority(&h->s_sc, cudaStreamNonBlocking, lo), "streams") &&
                       ck(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming), "events");
            for (auto *v : {&h->ev_bm, &h->ev_node, &h->ev_sc}) {
                v->assign(K, nullptr);
                for (auto &e : *v) sok = sok && ck(cudaEventCreateWithFlags(&e, cudaEventDisableTiming), "events");
            }
            if (!sok) return bail(LBM_ERR_CUDA, h->err);
            h->n_slab = K;
            h->ibp.order = h->node_order;
        }
    }
    if (ns && !h->n_slab) {
        // band entries that are first-layer cells of a 0D boundary (their pulls
        // may read ghosts, and the ghost kernel reads their force density)
        std::vector<uint8_t> xf((size_t)n, 0);
        for (int32_t c : L.lk_xf) xf[(size_t)c] = 1;
        std::vector<int32_t> ind, dep;
        for (int32_t c : L.band) ((L.flags[(size_t)c] & FL_XF) || xf[(size_t)c] ? dep : ind).push_back(c);
        int lo = 0, hi = 0;
        bool sok = ck(upload(h, &h->band_ind, ind), "band") && ck(upload(h, &h->band_dep, dep), "band") &&
                   ck(cudaDeviceGetStreamPriorityRange(&lo, &hi), "stream priorities") &&
                   ck(cudaStreamCreateWithPriority(&h->s_band, cudaStreamNonBlocking, lo), "streams") &&
                   ck(cudaStreamCreateWithPriority(&h->s_bc, cudaStreamNonBlocking, hi), "streams");
        for (auto *e : {&h->ev_ofork, &h->ev_oband, &h->ev_obc})
            sok = sok && ck(cudaEventCreateWithFlags(e, cudaEventDisableTiming), "events");
        if (!sok) return bail(LBM_ERR_CUDA, h->err);
        h->n_band_ind = (int)ind.size();
        h->n_band_dep = (int)dep.size();
        h->overlap = true;
    }
    if (!ck(set_up_small(h), "small-lattice tables")) return bail(LBM_ERR_CUDA, h->err);
    // A part needs cells: its stream-collide advances its step counter, the first
    // part's the lattice's.  Instances without cells have no boundaries either and
    // fall to the part before them (the first ones to the first part).
    std::vector<size_t> filled;
    for (size_t q = 0; q < L.inst.size(); q++)
        if (L.inst_cell_end[q] > L.inst_cell_begin[q]) filled.push_back(q);
    if (!ns && !h->small_blocks && filled.size() > 1) {
        const int K = (int)std::min<size_t>(filled.size(), lbm_handle::MAX_PARTS);
        int lo = 0, hi = 0;
        if (!(ck(dalloc(h, &h->step_parts, K), "step") &&
              ck(cudaDeviceGetStreamPriorityRange(&lo, &hi), "stream priorities") &&
              ck(cudaEventCreateWithFlags(&h->ev_parts, cudaEventDisableTiming), "events")))
            return bail(LBM_ERR_CUDA, h->err);
        h->parts.reserve(K);
        h->part_steps = std::min(16, h->graph_steps);
        while (h->graph_steps % h->part_steps || h->part_steps % 2) h->part_steps++;
        size_t m = 0;  // part k: the filled instances [m, e), its end where about k + 1 of K cells are
        for (int k = 0; k < K; k++) {
            size_t e = m + 1;
            auto off = [&](size_t q) { return std::llabs(K * L.inst_cell_end[filled[q - 1]] - (k + 1) * (int64_t)n); };
            while (e + (K - 1 - k) < filled.size() && off(e + 1) < off(e)) e++;
            if (k == K - 1) e = filled.size();
            const size_t q0 = m ? filled[m] : 0, q1 = e < filled.size() ? filled[e] : L.inst.size();
            h->parts.emplace_back();
            lbm_handle::Part &a = h->parts.back();
            a.c0 = (int)L.inst_cell_begin[q0];
            a.c1 = (int)L.inst_cell_end[q1 - 1];
            a.kp = h->kp;
            a.bp = h->bp;
            a.bp.priority = hi;
            a.bp.bc0 = L.inst[q0].bc_first;
            const int b1 = L.inst[q1 - 1].bc_first + L.inst[q1 - 1].n_bc;
            a.bp.n_bc = b1 - a.bp.bc0;
            auto at = [](const std::vector<int32_t> &v, int bc) {
                return (int)(std::lower_bound(v.begin(), v.end(), bc) - v.begin());
            };
            const int r0 = at(L.red_bc, a.bp.bc0), a0 = at(L.app_bc, a.bp.bc0);
            a.bp.n_red_blocks = at(L.red_bc, b1) - r0;
            a.bp.n_app_blocks = at(L.app_bc, b1) - a0;
            a.bp.red_bc += r0;
            a.bp.red_chunk += r0;
            a.bp.app_bc += a0;
            a.bp.app_chunk += a0;
            if (k) {
                a.kp.step = h->step_parts + k;
                if (!(ck(cudaStreamCreateWithFlags(&a.stream, cudaStreamNonBlocking), "streams") &&
                      ck(cudaEventCreateWithFlags(&a.done, cudaEventDisableTiming), "events")))
                    return bail(LBM_ERR_CUDA, h->err);
            }
            m = e;
        }
    }
    // Shape of stream-collide, unless the caller sets or tunes one: 16-bit batches
    // that exceed the L2 take 32 registers and more warps (96 uneven tubes FP16 348 ->
    // 334 us per step, 48: 161.2 -> 154.6, 24 equal ones 112.5 -> 110.7; a single tube
    // is no faster, a lattice with wall nodes slower, 183.5 -> 189.9), FP64 without wall
    // nodes 48 registers, which halves its spills (64 tubes 211.7 -> 210.9, a tube of 1.4 M
    // cells 338.7 -> 334.9; the aorta is slower, 2,205 -> 2,247).
    if (h->prec == LBM_F64) h->variant = ns ? 0 : 2;
    else if (h->sbytes == 2 && one_exceeds && !h->parts.empty()) h->variant = 1;
    if (h->ibp.n_fil && !(ck(cudaStreamCreateWithFlags(&h->s_fil, cudaStreamNonBlocking), "streams") &&
                          ck(cudaEventCreateWithFlags(&h->ev_nodes, cudaEventDisableTiming), "events") &&
                          ck(cudaEventCreateWithFlags(&h->ev_fil, cudaEventDisableTiming), "events")))
        return bail(LBM_ERR_CUDA, h->err);
    if (cudaDeviceSynchronize() != cudaSuccess) return bail(LBM_ERR_CUDA, "set-up failed");
    *out = h;
    return LBM_OK;
}

lbm_status lbm_set_0d_params(lbm_handle *h, int inst, int bc, const double *p, int np) {
    if (bad_inst(h, inst)) return fail(h, LBM_ERR_ARG, "bad instance");
    const InstParam &ip = h->L.inst[inst];
    if (bc < 0 || bc >= ip.n_bc || !p || np < 1 || np > 8) return fail(h, LBM_ERR_ARG, "bad boundary or params");
    BcParam &bp = h->L.bc[ip.bc_first + bc];
    if (const char *why = bad_params(bp, p, np)) return fail(h, LBM_ERR_ARG, why);
    for (int k = 0; k < np; k++) bp.par[k] = p[k];
    CK(h, cudaSetDevice(h->device));
    if (!h->par_ring) {
        CK(h, cudaHostAlloc((void **)&h->par_ring, lbm_handle::PAR_RING * sizeof(BcParam), cudaHostAllocMapped));
        CK(h, cudaHostGetDevicePointer((void **)&h->par_ring_dev, h->par_ring, 0));
        for (int k = 0; k < lbm_handle::PAR_RING; k++)
            CK(h, cudaEventCreateWithFlags(&h->par_ev[k], cudaEventDisableTiming));
    }
    const int slot = h->par_pos++ % lbm_handle::PAR_RING;
    CK(h, cudaEventSynchronize(h->par_ev[slot]));  // the copy that last used this slot has run
    h->par_ring[slot] = bp;
    CK(h, launch_copy_words(&h->par_ring_dev[slot], &h->bc_par[ip.bc_first + bc], sizeof(BcParam), h->stream));
    CK(h, cudaEventRecord(h->par_ev[slot], h->stream));
    return LBM_OK;
}

lbm_status lbm_read_0d_state_async(lbm_handle *h, int inst, double *out) {
    if (bad_inst(h, inst) || !out) return fail(h, LBM_ERR_ARG, "bad instance or array");
    const InstParam &ip = h->L.inst[inst];
    if (ip.n_bc == 0) return LBM_OK;
    CK(h, cudaSetDevice(h->device));
    // page-locked host memory that the device can address: the kernel writes
    // the rows there itself; otherwise through a device buffer and a copy
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, out) == cudaSuccess && at.type == cudaMemoryTypeHost && at.devicePointer) {
        CK(h, launch_state_rows(h->bc_state, h->bc_par, h->etab, ip.bc_first, ip.n_bc, (int)h->L.bc.size(),
                                (long long)h->steps, static_cast<double *>(at.devicePointer), h->stream));
        return LBM_OK;
    }
    (void)cudaGetLastError();
    if (!h->state_rows) CK(h, dalloc(h, &h->state_rows, 8 * std::max<size_t>(1, h->L.bc.size())));
    double *rows = h->state_rows + 8 * (size_t)ip.bc_first;
    CK(h, launch_state_rows(h->bc_state, h->bc_par, h->etab, ip.bc_first, ip.n_bc, (int)h->L.bc.size(),
                            (long long)h->steps, rows, h->stream));
    CK(h, cudaMemcpyAsync(out, rows, 8 * (size_t)ip.n_bc * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    return LBM_OK;
}

lbm_status lbm_init_populations(lbm_handle *h, int inst, const double *f) {
    if (bad_inst(h, inst) || !f) return fail(h, LBM_ERR_ARG, "bad instance or array");
    CK(h, cudaSetDevice(h->device));
    const Layout &L = h->L;
    const int64_t c0 = L.inst_cell_begin[inst], c1 = L.inst_cell_end[inst];
    const size_t M = (size_t)(c1 - c0);
    const lbm_instance_desc &d = h->inst[inst];
    const size_t nbox = (size_t)d.nx * d.ny * d.nz;
    std::vector<double> host(NQ * M);
    for (int i = 0; i < NQ; i++)
        for (size_t k = 0; k < M; k++) host[i * M + k] = f[i * nbox + (size_t)L.cell_box[c0 + k]];
    double *dev = nullptr;
    CK(h, cudaStreamSynchronize(h->stream));
    CK(h, cudaMalloc(&dev, host.size() * sizeof(double)));
    cudaError_t e = cudaMemcpy(dev, host.data(), host.size() * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = launch_init(h->prec, h->f[h->parity], h->kp, dev, (int)c0, (int)c1, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    cudaFree(dev);
    CK(h, e);
    return LBM_OK;
}

lbm_status lbm_step(lbm_handle *h, int64_t n) {
    if (!h || n < 0) return fail(h, LBM_ERR_ARG, "bad step count");
    CK(h, cudaSetDevice(h->device));
    if (h->timing) {
        for (int64_t k = 0; k < n; k++) {
            lbm_status s = launch_step(h, true);
            if (s != LBM_OK) return s;
            h->steps++;
        }
        return LBM_OK;
    }
    if (h->small_blocks && h->small_on && n >= h->small_from) return small_steps(h, n);
    int64_t left = n;
    const int per = h->parts.empty() ? h->graph_steps : h->part_steps;
    const bool use_short = n % per >= 3 * lbm_handle::SHORT_STEPS;
    while (left > 0) {
        const int len = left >= per ? per : use_short && left >= lbm_handle::SHORT_STEPS ? lbm_handle::SHORT_STEPS : 1;
        cudaGraphExec_t *graph = len == per ? h->graph : len == 1 ? h->graph1 : h->graph_short;
        lbm_status s = ensure_graph(h, graph, len);
        if (s != LBM_OK) return s;
        CK(h, cudaGraphLaunch(graph[h->parity], h->stream));
        if (len & 1) h->parity ^= 1;
        left -= len;
        h->steps += len;
    }
    return LBM_OK;
}

lbm_status lbm_step_io(lbm_handle *h, int inst, int bc, int64_t n, const double *params, int np, double *states) {
    if (bad_inst(h, inst)) return fail(h, LBM_ERR_ARG, "bad instance");
    const InstParam &ip = h->L.inst[inst];
    if (bc < 0 || bc >= ip.n_bc || !params || !states || np < 1 || np > 8 || n < 0)
        return fail(h, LBM_ERR_ARG, "bad boundary, step count, params or state array");
    if (n == 0) return LBM_OK;
    const int b = ip.bc_first + bc;
    BcParam &bp = h->L.bc[b];
    for (int64_t k = 0; k < n; k++)
        if (const char *why = bad_params(bp, params + k * np, np)) return fail(h, LBM_ERR_ARG, why);
    CK(h, cudaSetDevice(h->device));
    // both arrays must be page-locked host memory with a device address
    const double *pdev = nullptr;
    double *sdev = nullptr;
    {
        cudaPointerAttributes a{}, c{};
        if (cudaPointerGetAttributes(&a, params) != cudaSuccess || a.type != cudaMemoryTypeHost || !a.devicePointer ||
            cudaPointerGetAttributes(&c, states) != cudaSuccess || c.type != cudaMemoryTypeHost || !c.devicePointer) {
            (void)cudaGetLastError();
            return fail(h, LBM_ERR_ARG, "params and states must be page-locked host memory the device can address");
        }
        pdev = static_cast<const double *>(a.devicePointer);
        sdev = static_cast<double *>(c.devicePointer);
    }
    if (h->small_blocks && h->small_on && !h->timing) {
        SmallKParams sp = h->small;
        sp.io_params = pdev;
        sp.io_states = sdev;
        sp.io_np = np;
        sp.io_b = b;
        sp.io_b0 = ip.bc_first;
        sp.io_nb = ip.n_bc;
        const lbm_status st = small_steps(h, n, &sp);
        if (st != LBM_OK) return st;
        for (int k = 0; k < np; k++) bp.par[k] = params[(n - 1) * np + k];  // the host copy: the last set
        return LBM_OK;
    }
    if (!h->io_cursor) CK(h, dalloc(h, &h->io_cursor, 1));
    if (h->bp.cluster) CK(h, launch_io_base(h->step_dev, h->io_cursor, h->stream));
    else CK(h, cudaMemsetAsync(h->io_cursor, 0, sizeof(long long), h->stream));
    if (h->timing) {
        for (int64_t k = 0; k < n; k++) {
            lbm_status s = launch_io_step(h, pdev, np, b, sdev, inst, true, false, false);
            if (s != LBM_OK) return s;
            h->steps++;
        }
    } else {
        int64_t left = n;
        while (left > 0) {
            const int len = (int)std::min<int64_t>(left, h->graph_steps);
            cudaGraphExec_t g = nullptr;
            lbm_status s = ensure_io_graph(h, pdev, np, b, sdev, inst, len, &g);
            if (s != LBM_OK) return s;
            CK(h, cudaGraphLaunch(g, h->stream));
            if (len & 1) h->parity ^= 1;
            h->steps += len;
            left -= len;
        }
    }
    for (int k = 0; k < np; k++) bp.par[k] = params[(n - 1) * np + k];  // the host copy: the last set
    return LBM_OK;
}

lbm_status lbm_sync(lbm_handle *h) {
    if (!h) return LBM_ERR_ARG;
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    unsigned s = 0;
    CK(h, cudaMemcpy(&s, h->status, sizeof s, cudaMemcpyDeviceToHost));
    // before the others: blocks that went on alone may have made the lattice unstable
    if (s & 4u) return fail(h, LBM_ERR_CUDA, "the blocks of a multi-step kernel did not meet in time");
    if (s & 1u) return fail(h, LBM_ERR_UNSTABLE, "NaN/Inf or |v| > 0.3 in the lattice");
    if (s & 2u) return fail(h, LBM_ERR_UNSTABLE, "a wall node moved outside its immersed-boundary band");
    return LBM_OK;
}

lbm_status lbm_read_fields(lbm_handle *h, int inst, double *P, double *jx, double *jy, double *jz) {
    if (bad_inst(h, inst) || !P || !jx || !jy || !jz) return fail(h, LBM_ERR_ARG, "bad instance or array");
    CK(h, cudaSetDevice(h->device));
    lbm_status s = read_gather(h, inst, false);
    if (s != LBM_OK) return s;
    const Layout &L = h->L;
    const int64_t c0 = L.inst_cell_begin[inst], c1 = L.inst_cell_end[inst];
    const size_t M = (size_t)(c1 - c0);
    std::vector<double> mac(4 * M);
    const lbm_instance_desc &d = h->inst[inst];
    const size_t nbox = (size_t)d.nx * d.ny * d.nz;
    double *outs[4] = {P, jx, jy, jz};
    for (double *o : outs) std::fill(o, o + nbox, 0.0);  // while the GPU finishes
    CK(h, cudaStreamSynchronize(h->stream));
    CK(h, cudaMemcpy(mac.data(), h->rd_mac, 4 * M * sizeof(double), cudaMemcpyDeviceToHost));
    for (int k = 0; k < 4; k++) {
        for (size_t m = 0; m < M; m++) outs[k][L.cell_box[c0 + m]] = mac[k * M + m];
    }
    return LBM_OK;
}

lbm_status lbm_read_fields_device(lbm_handle *h, int inst, float *P, float *jx, float *jy, float *jz) {
    if (bad_inst(h, inst) || !P || !jx || !jy || !jz) return fail(h, LBM_ERR_ARG, "bad instance or array");
    CK(h, cudaSetDevice(h->device));
    const lbm_instance_desc &d = h->inst[inst];
    CK(h, launch_fields_box(h->prec, h->f[h->parity], h->kp, h->rowid + h->L.inst[inst].rowid_off, d.nx,
                            (int64_t)d.nx * d.ny * d.nz, P, jx, jy, jz, h->stream));
    return LBM_OK;
}

lbm_status lbm_read_populations(lbm_handle *h, int inst, double *f) {
    if (bad_inst(h, inst) || !f) return fail(h, LBM_ERR_ARG, "bad instance or array");
    CK(h, cudaSetDevice(h->device));
    lbm_status s = read_gather(h, inst, true);
    if (s != LBM_OK) return s;
    const Layout &L = h->L;
    const int64_t c0 = L.inst_cell_begin[inst], c1 = L.inst_cell_end[inst];
    const size_t M = (size_t)(c1 - c0);
    const lbm_instance_desc &d = h->inst[inst];
    const size_t nbox = (size_t)d.nx * d.ny * d.nz;
    std::vector<double> tmp(M);
    std::fill(f, f + NQ * nbox, 0.0);  // while the GPU finishes
    CK(h, cudaStreamSynchronize(h->stream));
    for (int i = 0; i < NQ; i++) {
        CK(h, cudaMemcpy(tmp.data(), h->rd_f19 + i * M, M * sizeof(double), cudaMemcpyDeviceToHost));
        double *o = f + i * nbox;
        for (size_t m = 0; m < M; m++) o[L.cell_box[c0 + m]] = tmp[m];
    }
    return LBM_OK;
}

lbm_status lbm_read_0d_state(lbm_handle *h, int inst, int bc, double *out) {
    if (bad_inst(h, inst) || !out) return fail(h, LBM_ERR_ARG, "bad instance or array");
    const InstParam &ip = h->L.inst[inst];
    if (bc < 0 || bc >= ip.n_bc) return fail(h, LBM_ERR_ARG, "bad boundary");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    BcState s;
    const size_t slot = (size_t)(h->steps & 1) * h->L.bc.size() + ip.bc_first + bc;  // state of t_steps
    CK(h, cudaMemcpy(&s, h->bc_state + slot, sizeof s, cudaMemcpyDeviceToHost));
    const BcParam &bp = h->L.bc[ip.bc_first + bc];
    out[0] = (double)h->steps;
    out[1] = s.Q;
    out[2] = s.Qu;
    out[3] = s.Pbar - 1.0 / 3.0;
    out[4] = bp.kind == BC_RCR ? s.Pw : (bp.kind == BC_LV ? s.Pv : s.Pstar_gauge);
    out[5] = 0.0;
    if (bp.kind == BC_LV) out[5] = s.Pv / h->L.etab[2 * (bp.etab_off + (int)(h->steps % bp.period))];
    out[6] = s.valve_open;
    out[7] = s.Td;
    return LBM_OK;
}

lbm_status lbm_read_waveforms(lbm_handle *h, int inst, double *out, int64_t max_rows, int64_t *rows) {
    if (bad_inst(h, inst) || !out || !rows || max_rows < 0) return fail(h, LBM_ERR_ARG, "bad arguments");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    const InstParam &ip = h->L.inst[inst];
    const int nb = (int)h->L.bc.size();
    const int64_t have = std::min<int64_t>({h->steps, (int64_t)h->wave_cap, max_rows});
    *rows = have;
    if (have == 0) return LBM_OK;
    std::vector<double> all((size_t)h->wave_cap * std::max(nb, 1) * 4, 0.0);
    if (nb > 0) CK(h, cudaMemcpy(all.data(), h->wave, all.size() * sizeof(double), cudaMemcpyDeviceToHost));
    const int width = 1 + 4 * ip.n_bc;
    for (int64_t r = 0; r < have; r++) {
        const int64_t stepno = h->steps - have + r;
        const size_t slot = (size_t)(stepno % h->wave_cap);
        double *row = out + r * width;
        row[0] = (double)stepno;
        for (int k = 0; k < ip.n_bc; k++)
            for (int m = 0; m < 4; m++) row[1 + 4 * k + m] = all[(slot * nb + ip.bc_first + k) * 4 + m];
    }
    return LBM_OK;
}

lbm_status lbm_read_ib(lbm_handle *h, int inst, double *X, double *Vs, double *F, double *Vf) {
    if (bad_inst(h, inst)) return fail(h, LBM_ERR_ARG, "bad instance");
    const InstParam &ip = h->L.inst[inst];
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    double *dst[4] = {X, Vs, F, Vf};
    const size_t m = 3 * (size_t)ip.n_ib, o = 3 * (size_t)ip.ib_off;
    if (h->prec == LBM_F64) {
        double *src[4] = {h->ibX, h->ibVs, h->ibF, h->ibVf};
        for (int k = 0; k < 4; k++)
            if (dst[k] && m) CK(h, cudaMemcpy(dst[k], src[k] + o, m * sizeof(double), cudaMemcpyDeviceToHost));
        return LBM_OK;
    }
    // FP32 node state; positions are X0 + D
    float *src[4] = {h->ibD32, h->ibVs32, h->ibF32, h->ibVf32};
    std::vector<float> tmp(m);
    for (int k = 0; k < 4; k++) {
        if (!dst[k] || !m) continue;
        CK(h, cudaMemcpy(tmp.data(), src[k] + o, m * sizeof(float), cudaMemcpyDeviceToHost));
        for (size_t j = 0; j < m; j++) dst[k][j] = (k == 0 ? h->L.ib_X0[o + j] : 0.0) + (double)tmp[j];
    }
    return LBM_OK;
}

lbm_status lbm_set_ib_state(lbm_handle *h, int inst, const double *X, const double *Vs) {
    if (bad_inst(h, inst) || !X || !Vs) return fail(h, LBM_ERR_ARG, "bad arguments");
    const InstParam &ip = h->L.inst[inst];
    for (int64_t s = 0; s < 3LL * ip.n_ib; s++)
        if (!std::isfinite(X[s]) || !std::isfinite(Vs[s])) return fail(h, LBM_ERR_ARG, "non-finite wall state");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    const size_t m = 3 * (size_t)ip.n_ib, o = 3 * (size_t)ip.ib_off;
    if (m && h->prec == LBM_F64) {
        CK(h, cudaMemcpy(h->ibX + o, X, m * sizeof(double), cudaMemcpyHostToDevice));
        CK(h, cudaMemcpy(h->ibVs + o, Vs, m * sizeof(double), cudaMemcpyHostToDevice));
    } else if (m) {  // FP32 node state: displacements from X0
        std::vector<float> D(m), V(m);
        for (size_t j = 0; j < m; j++) {
            D[j] = (float)(X[j] - h->L.ib_X0[o + j]);
            V[j] = (float)Vs[j];
        }
        CK(h, cudaMemcpy(h->ibD32 + o, D.data(), m * sizeof(float), cudaMemcpyHostToDevice));
        CK(h, cudaMemcpy(h->ibVs32 + o, V.data(), m * sizeof(float), cudaMemcpyHostToDevice));
    }
    return LBM_OK;
}

lbm_status lbm_set_multi_step(lbm_handle *h, int enable) {
    if (!h) return LBM_ERR_ARG;
    h->small_on = enable != 0;
    return LBM_OK;
}

lbm_status lbm_set_wait_limit(lbm_handle *h, int polls) {
    if (!h || polls < 1) return fail(h, LBM_ERR_ARG, "the limit must be at least 1 poll");
    h->small.polls = polls;
    return LBM_OK;
}

lbm_status lbm_set_kernel_timing(lbm_handle *h, int enable) {
    if (!h) return LBM_ERR_ARG;
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    if (enable && h->ev.empty()) {
        h->ev.resize(2048);
        for (auto &e : h->ev) CK(h, cudaEventCreate(&e));
    }
    h->timing = enable != 0;
    h->ev_used = 0;
    h->timed_launches = 0;
    h->timed_ms = 0.0;
    return LBM_OK;
}

lbm_status lbm_get_kernel_time(lbm_handle *h, int64_t *launches, double *total_ms) {
    if (!h || !launches || !total_ms) return fail(h, LBM_ERR_ARG, "bad arguments");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    for (size_t k = 0; k + 1 < h->ev_used; k += 2) {
        float ms = 0.f;
        CK(h, cudaEventElapsedTime(&ms, h->ev[k], h->ev[k + 1]));
        h->timed_ms += ms;
    }
    h->ev_used = 0;
    *launches = h->timed_launches;
    *total_ms = h->timed_ms;
    return LBM_OK;
}

lbm_status lbm_wall_shear(lbm_handle *h, int inst, double *wss) {
    if (bad_inst(h, inst) || !wss) return fail(h, LBM_ERR_ARG, "bad instance or array");
    CK(h, cudaSetDevice(h->device));
    const Layout &L = h->L;
    const int64_t c0 = L.inst_cell_begin[inst], c1 = L.inst_cell_end[inst];
    const size_t M = (size_t)(c1 - c0);
    if (!h->rd_mac) CK(h, dalloc(h, &h->rd_mac, 4 * (size_t)h->max_inst_cells));
    CK(h, launch_wall_shear(h->prec, h->f[h->parity], h->kp, (int)c0, (int)c1, h->rd_mac, h->stream));
    std::vector<double> tmp(3 * M);
    const lbm_instance_desc &d = h->inst[inst];
    const size_t nbox = (size_t)d.nx * d.ny * d.nz;
    std::fill(wss, wss + 3 * nbox, 0.0);  // while the GPU finishes
    CK(h, cudaMemcpyAsync(tmp.data(), h->rd_mac, 3 * M * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    for (size_t m = 0; m < M; m++)
        for (int a = 0; a < 3; a++) wss[3 * (size_t)L.cell_box[c0 + m] + a] = tmp[a * M + m];
    return LBM_OK;
}

lbm_status lbm_init_equilibrium(lbm_handle *h, int inst, const double *P, const double *vx, const double *vy,
                                const double *vz) {
    if (bad_inst(h, inst) || !P || !vx || !vy || !vz) return fail(h, LBM_ERR_ARG, "bad instance or array");
    CK(h, cudaSetDevice(h->device));
    const Layout &L = h->L;
    const int64_t c0 = L.inst_cell_begin[inst], c1 = L.inst_cell_end[inst];
    const size_t M = (size_t)(c1 - c0);
    const double *src[4] = {P, vx, vy, vz};
    std::vector<double> host(4 * M);
    for (int k = 0; k < 4; k++)
        for (size_t m = 0; m < M; m++) {
            const double v = src[k][(size_t)L.cell_box[c0 + m]];
            if ((L.flags[c0 + m] & FL_ACTIVE) && !std::isfinite(v)) return fail(h, LBM_ERR_ARG, "non-finite field value");
            host[k * M + m] = v;
        }
    if (!h->rd_mac) CK(h, dalloc(h, &h->rd_mac, 4 * (size_t)h->max_inst_cells));
    CK(h, cudaStreamSynchronize(h->stream));
    CK(h, cudaMemcpy(h->rd_mac, host.data(), host.size() * sizeof(double), cudaMemcpyHostToDevice));
    CK(h, launch_init_eq(h->prec, h->f[h->parity], h->kp, h->rd_mac, (int)c0, (int)c1, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

namespace {
struct CkptHeader {
    char magic[8];
    int64_t version, prec, n_stored, n_bc, n_ib, n_xf, wave_cap, steps, parity;
};
struct CkptSection {  // rows of row_bytes on the device, pitch apart; packed in the checkpoint
    void *dev;
    size_t row_bytes, rows = 1, pitch = 0;
    size_t bytes() const { return row_bytes * rows; }
    // one row by a plain copy: the documented limit of a pitch (cudaDevAttrMaxPitch, 2^31 - 1) is
    // less than the force density of a large FP64 lattice or a long waveform ring; a direction's
    // row stays below it
    cudaError_t copy(void *packed, bool save) const {
        if (rows == 1)
            return save ? cudaMemcpy(packed, dev, row_bytes, cudaMemcpyDeviceToHost)
                        : cudaMemcpy(dev, packed, row_bytes, cudaMemcpyHostToDevice);
        return save ? cudaMemcpy2D(packed, row_bytes, dev, pitch, row_bytes, rows, cudaMemcpyDeviceToHost)
                    : cudaMemcpy2D(dev, pitch, packed, row_bytes, row_bytes, rows, cudaMemcpyHostToDevice);
    }
};
std::vector<CkptSection> ckpt_sections(lbm_handle *h) {
    const Layout &L = h->L;
    const size_t n = (size_t)L.n_stored, nb = L.bc.size(), ns = L.ib_dA.size();
    std::vector<CkptSection> v = {
        {h->f[h->parity], n * (size_t)h->sbytes, NQ, (size_t)population_cells((int64_t)n) * h->sbytes},
        {h->b, 4 * n * (size_t)h->rbytes},
        {h->bc_state, 2 * std::max<size_t>(nb, 1) * sizeof(BcState)},
        {h->v0, 3 * std::max<size_t>(1, L.xf.size()) * sizeof(double)},
        {h->wave, (size_t)h->wave_cap * std::max<size_t>(1, nb) * 4 * sizeof(double)},
        {h->step_dev, sizeof(long long)},
        {h->status, sizeof(unsigned)},
    };
    if (ns) {
        if (h->prec == LBM_F64) {
            double *ib[5] = {h->ibX, h->ibVs, h->ibI, h->ibF, h->ibVf};
            for (double *a : ib) v.push_back({a, 3 * ns * sizeof(double)});
        } else {
            float *ib[5] = {h->ibD32, h->ibVs32, h->ibI32, h->ibF32, h->ibVf32};
            for (float *a : ib) v.push_back({a, 3 * ns * sizeof(float)});
        }
    }
    return v;
}
CkptHeader ckpt_header(const lbm_handle *h) {
    CkptHeader hd;
    memset(&hd, 0, sizeof hd);
    memcpy(hd.magic, "LBMCKPT1", 8);
    hd.version = 1;
    hd.prec = h->prec;
    hd.n_stored = h->L.n_stored;
    hd.n_bc = (int64_t)h->L.bc.size();
    hd.n_ib = (int64_t)h->L.ib_dA.size();
    hd.n_xf = (int64_t)h->L.xf.size();
    hd.wave_cap = h->wave_cap;
    hd.steps = h->steps;
    hd.parity = h->parity;
    return hd;
}
}  // namespace

lbm_status lbm_checkpoint_size(lbm_handle *h, int64_t *bytes) {
    if (!h || !bytes) return fail(h, LBM_ERR_ARG, "bad arguments");
    size_t total = sizeof(CkptHeader);
    for (auto &sct : ckpt_sections(h)) total += sct.bytes();
    *bytes = (int64_t)total;
    return LBM_OK;
}

lbm_status lbm_checkpoint_save(lbm_handle *h, void *buf, int64_t bytes) {
    int64_t need = 0;
    if (!h || !buf || lbm_checkpoint_size(h, &need) != LBM_OK || bytes < need)
        return fail(h, LBM_ERR_ARG, "null buffer or smaller than lbm_checkpoint_size");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    uint8_t *p = static_cast<uint8_t *>(buf);
    const CkptHeader hd = ckpt_header(h);
    memcpy(p, &hd, sizeof hd);
    p += sizeof hd;
    for (auto &sct : ckpt_sections(h)) {
        if (sct.bytes()) CK(h, sct.copy(p, true));
        p += sct.bytes();
    }
    return LBM_OK;
}

lbm_status lbm_checkpoint_load(lbm_handle *h, const void *buf, int64_t bytes) {
    int64_t need = 0;
    if (!h || !buf || lbm_checkpoint_size(h, &need) != LBM_OK || bytes < need)
        return fail(h, LBM_ERR_ARG, "null buffer or smaller than lbm_checkpoint_size");
    CkptHeader hd, mine = ckpt_header(h);
    memcpy(&hd, buf, sizeof hd);
    if (memcmp(hd.magic, mine.magic, 8) != 0 || hd.version != mine.version || hd.prec != mine.prec ||
        hd.n_stored != mine.n_stored || hd.n_bc != mine.n_bc || hd.n_ib != mine.n_ib || hd.n_xf != mine.n_xf ||
        hd.wave_cap != mine.wave_cap || (hd.parity != 0 && hd.parity != 1) || hd.steps < 0)
        return fail(h, LBM_ERR_ARG, "checkpoint does not match this handle's configuration");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    h->parity = (int)hd.parity;  // selects the resident buffer the sections refer to
    h->steps = hd.steps;
    const uint8_t *p = static_cast<const uint8_t *>(buf) + sizeof hd;
    for (auto &sct : ckpt_sections(h)) {
        if (sct.bytes()) CK(h, sct.copy(const_cast<uint8_t *>(p), false));
        p += sct.bytes();
    }
    return LBM_OK;
}

lbm_status lbm_set_0d_state(lbm_handle *h, int inst, int bc, const double *s3) {
    if (bad_inst(h, inst) || !s3) return fail(h, LBM_ERR_ARG, "bad instance or array");
    const InstParam &ip = h->L.inst[inst];
    if (bc < 0 || bc >= ip.n_bc) return fail(h, LBM_ERR_ARG, "bad boundary");
    if (!std::isfinite(s3[0]) || !(s3[1] == 0.0 || s3[1] == 1.0)) return fail(h, LBM_ERR_ARG, "bad 0D state");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    const size_t slot = (size_t)(h->steps & 1) * h->L.bc.size() + ip.bc_first + bc;
    BcState st;
    CK(h, cudaMemcpy(&st, h->bc_state + slot, sizeof st, cudaMemcpyDeviceToHost));
    const BcParam &bp = h->L.bc[ip.bc_first + bc];
    if (bp.kind == BC_RCR) st.Pw = s3[0];
    if (bp.kind == BC_LV) st.Pv = s3[0];
    st.valve_open = s3[1];
    st.Td = s3[2];
    CK(h, cudaMemcpy(h->bc_state + slot, &st, sizeof st, cudaMemcpyHostToDevice));
    return LBM_OK;
}

lbm_status lbm_cycle_change(lbm_handle *h, const int64_t *period, double *delta) {
    if (!h || !period || !delta) return fail(h, LBM_ERR_ARG, "bad arguments");
    const int ni = (int)h->inst.size();
    std::vector<long long> per(ni);
    for (int q = 0; q < ni; q++) {
        if (period[q] < 1 || 2 * period[q] > h->wave_cap)
            return fail(h, LBM_ERR_ARG, "period must be >= 1 and two periods must fit the waveform capacity");
        per[q] = 2 * period[q] > h->steps ? 0 : period[q];  // 0: not enough history yet, delta = -1
    }
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaMemcpyAsync(h->inst_period, per.data(), ni * sizeof(long long), cudaMemcpyHostToDevice, h->stream));
    CK(h, launch_cycle_change(h->bp, h->inst_bc, h->inst_bc + ni, h->inst_period, (long long)h->steps, h->inst_delta,
                              ni, h->stream));
    CK(h, cudaMemcpyAsync(delta, h->inst_delta, ni * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

lbm_status lbm_set_stream_collide_shape(lbm_handle *h, int block, int variant) {
    if (!h || block < 32 || block > 256 || (block % 32) != 0 || variant < 0 || variant >= SC_VARIANTS)
        return fail(h, LBM_ERR_ARG, "block must be a multiple of 32 in [32, 256], variant in [0, 4]");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    if (block != h->block || variant != h->variant) drop_graphs(h);
    h->block = block;
    h->variant = variant;
    return LBM_OK;
}

lbm_status lbm_autotune(lbm_handle *h, int iters, int *block, int *min_blocks, int *cells_per_thread,
                        double *times_ms) {
    if (!h || iters < 1 || !block || !min_blocks || !cells_per_thread) return fail(h, LBM_ERR_ARG, "bad arguments");
    CK(h, cudaSetDevice(h->device));
    CK(h, cudaStreamSynchronize(h->stream));
    KParams kp = h->kp;
    kp.step = nullptr;  // timing launches must not advance the step index
    void *fin = h->f[h->parity], *fout = h->f[1 - h->parity];
    const bool whole_steps = !h->ibp.n_nodes;
    TuneScratch scratch;
    if (whole_steps) {
        const lbm_status s = tune_scratch(h, scratch);
        if (s != LBM_OK) return s;
    }
    const int len = std::min(iters, 32), reps = (iters + len - 1) / len;
    cudaEvent_t e0, e1;
    CK(h, cudaEventCreate(&e0));
    CK(h, cudaEventCreate(&e1));
    static const int blocks[4] = {64, 128, 192, 256};
    float best = 1e30f;
    int bb = h->block, bv = h->variant;
    for (int v = 0; v < SC_VARIANTS; v++)
        for (int bi = 0; bi < 4; bi++) {
            float ms = 0.f;
            if (whole_steps) {
                const lbm_status s = tune_candidate(h, scratch, blocks[bi], v, len, reps, e0, e1, &ms);
                if (s != LBM_OK) {
                    cudaEventDestroy(e0);
                    cudaEventDestroy(e1);
                    return s;
                }
            } else {
                CK(h, launch_stream_collide(h->prec, fin, fout, kp, blocks[bi], v, h->stream));  // warm-up
                CK(h, cudaEventRecord(e0, h->stream));
                for (int k = 0; k < iters; k++)
                    CK(h, launch_stream_collide(h->prec, fin, fout, kp, blocks[bi], v, h->stream));
                CK(h, cudaEventRecord(e1, h->stream));
                CK(h, cudaEventSynchronize(e1));
                CK(h, cudaEventElapsedTime(&ms, e0, e1));
                ms /= (float)iters;
            }
            if (times_ms) times_ms[4 * v + bi] = ms;
            if (ms < best) {
                best = ms;
                bb = blocks[bi];
                bv = v;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    // the timing launches wrote f* from the resident state into the other buffer,
    // which the next step overwrites; the resident state itself is unchanged
    if (bb != h->block || bv != h->variant) drop_graphs(h);
    h->block = bb;
    h->variant = bv;
    *block = bb;
    *min_blocks = stream_collide_min_blocks(bv);
    *cells_per_thread = stream_collide_cells_per_thread(bv);
    return LBM_OK;
}

lbm_status lbm_get_info(lbm_handle *h, lbm_info_t *info) {
    if (!h || !info) return LBM_ERR_ARG;
    info->fluid_cells = h->L.n_fluid;
    info->stored_cells = h->L.n_stored;
    info->box_cells = h->L.n_box;
    info->band_cells = (int64_t)h->L.band.size();
    info->ib_nodes = (int64_t)h->L.ib_dA.size();
    info->links = (int64_t)h->L.lk_xb.size();
    info->steps = h->steps;
    info->device_bytes = h->bytes;
    info->precision = h->prec;
    info->bytes_per_population = h->sbytes;
    info->slabs = h->n_slab;
    int n = 0;
    const Layout &L = h->L;
    if (h->n_slab) {
        for (int s = 0; s < h->n_slab; s++)
            n += (L.slab_band[s + 1] > L.slab_band[s]) + (L.slab_node[s + 1] > L.slab_node[s]) +
                 (L.slab_cell[s + 1] > L.slab_cell[s]);
    } else {
        n = (L.n_stored > 0) + (L.ib_dA.empty() ? 0 : (L.band.empty() ? 0 : 1) + 1 + (L.fil_start.empty() ? 0 : 1));
    }
    info->launches_per_step = n + (L.bc.empty() ? 0 : h->bp.cluster ? 1 : 2);
    info->launches_first_step = info->launches_per_step;
    if (h->overlap)  // band velocities as the two lists (an empty list launches nothing)
        info->launches_per_step += (h->n_band_ind > 0) + (h->n_band_dep > 0) - 1;
    info->graph_steps = h->parts.empty() ? h->graph_steps : h->part_steps;
    const bool multi = h->small_blocks && h->small_on;
    info->short_graph_steps = multi ? 0 : lbm_handle::SHORT_STEPS;
    info->parts = std::max(1, (int)h->parts.size());
    info->steps_per_launch = multi ? SMALL_MAX_STEPS : 0;
    info->multi_step_from = multi ? h->small_from : 0;
    return LBM_OK;
}

const char *lbm_last_error(const lbm_handle *h) { return h ? h->err.c_str() : "null handle"; }

void lbm_destroy(lbm_handle *h) {
    if (!h) return;
    cudaSetDevice(h->device);
    if (h->stream) cudaStreamSynchronize(h->stream);
    for (int k = 0; k < 2; k++) {
        if (h->graph[k]) cudaGraphExecDestroy(h->graph[k]);
        if (h->graph_short[k]) cudaGraphExecDestroy(h->graph_short[k]);
        if (h->graph1[k]) cudaGraphExecDestroy(h->graph1[k]);
    }
    for (auto &g : h->io_graphs) cudaGraphExecDestroy(g.exec);
    for (auto e : h->ev) cudaEventDestroy(e);
    for (auto *v : {&h->ev_bm, &h->ev_node, &h->ev_sc})
        for (auto e : *v)
            if (e) cudaEventDestroy(e);
    if (h->ev_fork) cudaEventDestroy(h->ev_fork);
    for (auto e : {h->ev_ofork, h->ev_oband, h->ev_obc, h->ev_nodes, h->ev_fil})
        if (e) cudaEventDestroy(e);
    if (h->s_fil) cudaStreamDestroy(h->s_fil);
    for (auto &a : h->parts) {
        if (a.stream) cudaStreamDestroy(a.stream);
        if (a.done) cudaEventDestroy(a.done);
    }
    if (h->ev_parts) cudaEventDestroy(h->ev_parts);
    if (h->s_band) cudaStreamDestroy(h->s_band);
    if (h->s_bc) cudaStreamDestroy(h->s_bc);
    if (h->s_node) cudaStreamDestroy(h->s_node);
    if (h->s_sc) cudaStreamDestroy(h->s_sc);
    if (h->par_ring) {
        for (auto e : h->par_ev) cudaEventDestroy(e);
        cudaFreeHost(h->par_ring);
    }
    for (void *p : h->allocs) cudaFree(p);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    delete h;
}

}  // extern "C"

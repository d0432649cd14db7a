// The 0D step of a boundary and the sums over its first layer, shared by the
// boundary kernels and the multi-step kernels of small lattices and grids.
#pragma once
#include "lbm_zero_d.cuh"

namespace lbm {

// The 0D step of boundary b from the sums over its first layer (taken by one
// thread): the state of t_{n+1} and, if store, the state and the waveform row
// written; returns what the ghost pass needs.
static __device__ BcStepResult bc_step(const BcParam &P, int b, double Q, double Ps, long long n,
                                       const BcKParams &q, bool store) {
    const BcState old = q.state[(size_t)(n & 1) * q.n_bc_total + b];
    int ptype, closed;
    double Sm;
    const double Psum = (double)P.n_xf / 3.0 + Ps;  // sum of P over the layer
    const BcState st = zero_d_step(P, old, Q, Psum, (double)P.n_xf, n, q.etab, &ptype, &closed, &Sm);
    if (store) {
        q.state[(size_t)((n + 1) & 1) * q.n_bc_total + b] = st;
        double *w = q.wave + ((size_t)(n % q.wave_cap) * q.n_bc_total + b) * 4;
        w[0] = st.Qu;
        w[1] = st.Pbar - 1.0 / 3.0;
        w[2] = (P.kind == BC_RCR) ? st.Pw : (P.kind == BC_LV ? st.Pv : st.Pstar_gauge);
        w[3] = st.valve_open;
    }
    BcStepResult r;
    r.Pg = st.Pstar_gauge;
    r.S = Sm;
    r.cosp = r.sinp = 0.0;
    if (P.kind == BC_VELOCITY) {  // the inlet's phase, once for every link of the boundary
        const double wv = P.par[0], tn1 = (double)(n + 1);
        r.cosp = cos(wv * tn1);
        r.sinp = sin(wv * tn1);
    }
    r.ptype = ptype;
    r.closed = closed;
    r.pad0 = r.pad1 = 0;
    return r;
}

// a / b, rounded to nearest, from inv_b = 1 / b rounded to nearest: Markstein's
// correction (P. Markstein, IBM J. Res. Dev. 34, 1990): with q within an ulp of
// a / b, q + (a - b q) inv_b is the correctly rounded quotient.  The first step
// brings a inv_b within an ulp.  Five dependent operations, half the latency of a
// division; magnitudes near the ends of the range are divided.
static __device__ __forceinline__ double quotient(double a, double b, double inv_b) {
    // binary exponents within +-500 of one (integer tests: an FP64 comparison waits as long as an addition)
    const unsigned ea = ((unsigned)__double2hiint(a) >> 20) & 0x7ffu, eb = ((unsigned)__double2hiint(b) >> 20) & 0x7ffu;
    if (ea - 523u > 1000u || eb - 823u > 400u) return a / b;
    double q = a * inv_b;
    q = fma(fma(-b, q, a), inv_b, q);
    return fma(fma(-b, q, a), inv_b, q);
}

// zero_d_step with forward Euler in two parts, in the same expressions: what
// does not depend on the step's flow, taken beside other work (an FP64 division
// is about 700 cycles on this part), and the rest.  boundary_euler: whether the
// boundary marches so.
struct Ahead {
    double p0_rc, inv_c; // RCR: P_w / (R_d C) and 1 / C
    double inv_cv, dcv;  // LV: 1 / C_v and dC_v/dt, C_v = 1/E
};
static __device__ __forceinline__ bool boundary_euler(const BcParam &P) {
    const int order = (int)P.par[4];
    return !((P.kind == BC_RCR || P.kind == BC_LV) && (order == 2 || order == 4));
}
static __device__ __forceinline__ void ahead_terms(const BcParam &P, const BcState &st, long long n, const double *etab,
                                                   Ahead *a) {
    if (P.kind == BC_RCR) {
        a->p0_rc = st.Pw / (P.par[2] * P.par[1]);
        a->inv_c = 1.0 / P.par[1];
    }
    if (P.kind == BC_LV) {
        const double E = etab[2 * (P.etab_off + (int)(n % P.period))];
        const double Ed = etab[2 * (P.etab_off + (int)(n % P.period)) + 1];
        const double Cv = 1.0 / E;
        a->dcv = -Ed / (E * E);
        a->inv_cv = 1.0 / Cv;
    }
}
// Q the flow, Qmean = Q / area and Pbar the mean pressure of the first layer
static __device__ __forceinline__ BcState zero_d_euler(const BcParam &P, const BcState &old, const Ahead &a, double Q,
                                                       double Qmean, double Pbar, long long n, int *ptype, int *closed,
                                                       double *Smooth) {
    BcState st = old;
    st.Q = Q;
    st.Qu = P.q_scale ? Qmean : Q;
    st.Pbar = Pbar;
    *ptype = 1;
    *closed = 0;
    *Smooth = 0.0;
    if (P.kind == BC_RCR) {
        const double Qout = -st.Qu;
        const double Pw = old.Pw + (quotient(Qout, P.par[1], a.inv_c) - a.p0_rc);
        st.Pw = Pw;
        st.Pstar_gauge = Pw + P.par[0] * Qout;
    } else if (P.kind == BC_PRESSURE) {
        st.Pstar_gauge = P.par[0];
    } else if (P.kind == BC_LV) {
        const double Qin = (old.valve_open != 0.0) ? st.Qu : 0.0;
        double Pv = old.Pv - a.inv_cv * (a.dcv * old.Pv + Qin);
        if (old.valve_open != 0.0) {
            if (st.Qu < 0.0) {  // closure: the inflow has reversed
                st.valve_open = 0.0;
                st.Td = (double)n;
                *closed = 1;
            }
        } else {
            if (Pv < P.par[1]) Pv = P.par[1];
            if (Pv > st.Pbar - 1.0 / 3.0) st.valve_open = 1.0;
        }
        st.Pv = Pv;
        st.Pstar_gauge = Pv;
        *ptype = st.valve_open != 0.0;
        if (!*ptype) *Smooth = smooth_to_zero((double)(n + 1), st.Td, P.par[2]);  // unused with the valve open
    } else {
        *ptype = 0;
    }
    return st;
}

// The partial sums of the first layer (n_red of them, 2 doubles each) added in
// the order of bc_sum_partials by the first warp: lane 0 gets the flow and lane
// 1 the pressure.
static __device__ __forceinline__ double sum_partials_pair(const double *part, int n_red) {
    const int lane = threadIdx.x & 31;
    if (n_red <= 8) {  // the butterfly's additions that are not of zeros, each lane its own quantity
        double a[8];
        a[0] = 0.0 + part[lane & 1];
        if (n_red > 1) {
#pragma unroll
            for (int k = 1; k < 8; k++) a[k] = k < n_red ? 0.0 + part[2 * k + (lane & 1)] : 0.0;
            if (n_red > 4)
#pragma unroll
                for (int k = 0; k < 4; k++) a[k] += a[k + 4];
            if (n_red > 2) {
                a[0] += a[2];
                a[1] += a[3];
            }
            a[0] += a[1];
        }
        return a[0];
    }
    double a = 0.0, c = 0.0;
    for (int k = lane; k < n_red; k += 32) {
        a += part[2 * k];
        c += part[2 * k + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    return (lane & 1) ? c : a;
}

// s / 3, rounded to nearest, by the same correction in the arithmetic type
static __device__ __forceinline__ float third_of(float s) {
    const unsigned e = (__float_as_uint(s) >> 23) & 0xffu;
    if (e - 40u > 200u) return s / 3.0f;
    const float q = s * (1.0f / 3.0f);
    const float q1 = fmaf(fmaf(-3.0f, q, s), 1.0f / 3.0f, q);
    return fmaf(fmaf(-3.0f, q1, s), 1.0f / 3.0f, q1);
}
static __device__ __forceinline__ double third_of(double s) { return quotient(s, 3.0, 1.0 / 3.0); }

// Sum of 256 values of shared memory by one warp, in the order of the tree of
// k_bc_reduce (128, 64, 32, then within the warp); lane 0 gets it.
static __device__ __forceinline__ double tree_256(const double *v) {
    v += threadIdx.x & 31;
    double a[4];
#pragma unroll
    for (int h = 0; h < 4; h++) a[h] = v[32 * h] + v[32 * (h + 4)];
    a[0] = (a[0] + a[2]) + (a[1] + a[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[0] += __shfl_down_sync(0xffffffffu, a[0], o);
    return a[0];
}

// the 8-value state row of a boundary after `steps` steps:
// {t, Q, Q_u, Pbar_gauge, state, C_v P_v (LV), valve_open, T_d}
__device__ __forceinline__ void state_row(const BcState &s, const BcParam &P, const double *etab, long long steps,
                                          double *o) {
    o[0] = (double)steps;
    o[1] = s.Q;
    o[2] = s.Qu;
    o[3] = s.Pbar - 1.0 / 3.0;
    o[4] = P.kind == BC_RCR ? s.Pw : (P.kind == BC_LV ? s.Pv : s.Pstar_gauge);
    o[5] = P.kind == BC_LV ? s.Pv / etab[2 * (P.etab_off + (int)(steps % P.period))] : 0.0;
    o[6] = s.valve_open;
    o[7] = s.Td;
}

}  // namespace lbm

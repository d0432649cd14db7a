// The 0D step of a boundary and the ghost populations it sets, shared by the
// boundary kernels and the multi-step kernel of small lattices.
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

// the velocity set for a direction known only at run time
static __constant__ signed char c_ex[NQ] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
static __constant__ signed char c_ey[NQ] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
static __constant__ signed char c_ez[NQ] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};

// f^eq_i(P + dP, vs) - f^eq_i(P, vf)
template <class R> __device__ __forceinline__ R feq_change(int i, R dP, const R vs[3], const R vf[3]) {
    const R ex = c_ex[i], ey = c_ey[i], ez = c_ez[i];
    const R w = i == 0 ? R(1.0 / 3.0) : (i < 7 ? R(1.0 / 18.0) : R(1.0 / 36.0));
    const R eus = ex * vs[0] + ey * vs[1] + ez * vs[2];
    const R euf = ex * vf[0] + ey * vf[1] + ez * vf[2];
    const R us2 = vs[0] * vs[0] + vs[1] * vs[1] + vs[2] * vs[2];
    const R uf2 = vf[0] * vf[0] + vf[1] * vf[1] + vf[2] * vf[2];
    return w * R(3) * dP + w * (R(3) * (eus - euf) + R(4.5) * (eus * eus - euf * euf) - R(1.5) * (us2 - uf2));
}

// f^eq_i(P*, v*) - f^eq_i(P(x_f), v(x_f)) of one link (Eq. Non-equilibrium3):
// vf the forced velocity and sdf the sum s at x_f, pr the inlet profile of the
// link's node (velocity kind), v0o the closure velocity of x_f (LV kind;
// rewritten at v0 when the valve closes in this step).
template <class R>
__device__ __forceinline__ R ghost_change(const BcParam &P, const BcStepResult &r, int i, const R vf[3], R sdf,
                                          const double pr[3], const double v0o[3], double *v0) {
    R dP, vs[3];  // P* - P(x_f) and v*
    if (r.ptype) {  // pressure-type: (P_0D(t_{n+1}), v(x_f, t_n))
        dP = (R)r.Pg - sdf / R(3);
        vs[0] = vf[0];
        vs[1] = vf[1];
        vs[2] = vf[2];
    } else {        // velocity-type: (P(x_f, t_n), v_0D(t_{n+1}))
        dP = R(0);
        vs[0] = vs[1] = vs[2] = R(0);
        if (P.kind == BC_VELOCITY) {
            vs[P.axis] = (R)((double)P.sign * (pr[0] + pr[1] * r.cosp - pr[2] * r.sinp));
        } else if (P.kind == BC_LV) {  // closed valve: v_0(T_d) S(t, T_d, N_S)
            R u0[3];
            if (r.closed) {  // v_0(T_d) = v(x_f, T_d); links sharing x_f store the same value
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    u0[a] = vf[a];
                    v0[a] = (double)vf[a];
                }
            } else {
#pragma unroll
                for (int a = 0; a < 3; a++) u0[a] = (R)v0o[a];
            }
            const R Sm = (R)r.S;
            vs[0] = u0[0] * Sm;
            vs[1] = u0[1] * Sm;
            vs[2] = u0[2] * Sm;
        }
    }
    return feq_change<R>(i, dP, vs, vf);
}

}  // namespace lbm

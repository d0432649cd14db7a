// The ghost populations that a boundary of the D3Q19 lattice sets, shared by the
// boundary kernels and the multi-step kernel of small lattices.  Apart from
// lbm_boundary.cuh because of the tables: every kernel of a module with
// __constant__ variables starts about 0.1 us later, also one that does not read
// them (the three kernels of an axisymmetric step 12.8 -> 13.1 us).
#pragma once
#include "lbm_boundary.cuh"

namespace lbm {

// the velocity set for a direction known only at run time
static __constant__ signed char c_ex[NQ] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
static __constant__ signed char c_ey[NQ] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
static __constant__ signed char c_ez[NQ] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};

// f^eq_i(P + dP, vs) - f^eq_i(P, vf), (ex, ey, ez) = e_i and w = w_i
template <class R> __device__ __forceinline__ R feq_change(R ex, R ey, R ez, R w, R dP, const R vs[3], const R vf[3]) {
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
    const R w = i == 0 ? R(1.0 / 3.0) : (i < 7 ? R(1.0 / 18.0) : R(1.0 / 36.0));
    return feq_change<R>((R)c_ex[i], (R)c_ey[i], (R)c_ez[i], w, dP, vs, vf);
}

}  // namespace lbm

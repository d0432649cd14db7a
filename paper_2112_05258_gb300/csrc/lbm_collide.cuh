// The collision of one cell (moments, equilibrium, Guo forcing, BGK), shared
// by the stream-collide kernel and the multi-step kernel of small lattices so
// that both give the same bits.
#pragma once
#include "lbm_device.cuh"

namespace lbm {

// out(i, c) is the address of population i of cell c; the moments of f come back.
// LARGE: the populations exceed the L2, and the stores stay there (keep_in_l2).
template <class R> struct Moments {
    R sd, jx, jy, jz;  // sum s, j
};
template <class S, class R, bool FORCED, bool LARGE, class Out>
__device__ __forceinline__ Moments<R> collide_store(const Out &out, const KParams &p, const R (&f)[NQ], R omega,
                                                    uint32_t fl, int c) {
    constexpr int NP = (NQ - 1) / 2;
    R Sp[NP], Dp[NP];
#pragma unroll
    for (int q = 0; q < NP; q++) {
        Sp[q] = f[2 * q + 1] + f[2 * q + 2];
        Dp[q] = f[2 * q + 1] - f[2 * q + 2];
    }
    R sd = f[0], jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int q = 0; q < NP; q++) {
        sd += Sp[q];
        const int i = 2 * q + 1;
        if (cx(i) > 0) jx += Dp[q];
        if (cx(i) < 0) jx -= Dp[q];
        if (cy(i) > 0) jy += Dp[q];
        if (cy(i) < 0) jy -= Dp[q];
        if (cz(i) > 0) jz += Dp[q];
        if (cz(i) < 0) jz -= Dp[q];
    }
    R bx = 0, by = 0, bz = 0;
    if (FORCED && (fl & FL_BAND)) {
        const typename Vec4<R>::T bb = static_cast<const typename Vec4<R>::T *>(p.b)[c];
        bx = bb.x;
        by = bb.y;
        bz = bb.z;
    }
    const R vx = FORCED ? jx + R(0.5) * bx : jx;
    const R vy = FORCED ? jy + R(0.5) * by : jy;
    const R vz = FORCED ? jz + R(0.5) * bz : jz;
    if (fl & FL_XF) {
        R *aux = static_cast<R *>(p.aux);
        const size_t N = (size_t)p.n;
        aux[c] = sd;
        aux[N + c] = jx;
        aux[2 * N + c] = jy;
        aux[3 * N + c] = jz;
    }
    const R vv = vx * vx + vy * vy + vz * vz;
    if (!(sd - sd == R(0)) || !(vv <= R(0.09))) atomicOr(p.status, 1u);

    const uint64_t keep = LARGE ? keep_in_l2(p.keep) : 0;
    auto put = [&](S *a, R v) {
        if (LARGE) st_keep(a, v, keep);
        else Storage<S>::st(a, v);
    };
    const R om1 = R(1) - omega;
    const R K = sd - R(1.5) * vv;
    // per weight class (1/18 faces, 1/36 edges): omega w K, 9/2 omega w, 3 omega w
    const R ow1 = omega * R(1.0 / 18.0), ow2 = omega * R(1.0 / 36.0);
    const R wK1 = ow1 * K, wK2 = ow2 * K;
    const R a1 = R(4.5) * ow1, a2 = R(4.5) * ow2;
    const R b1 = R(3) * ow1, b2 = R(3) * ow2;
    R kw1 = 0, kw2 = 0, vb = 0;
    if (FORCED) {
        const R kf = R(1) - R(0.5) * omega;
        kw1 = kf * R(1.0 / 18.0);
        kw2 = kf * R(1.0 / 36.0);
        vb = vx * bx + vy * by + vz * bz;
    }
    R post0 = om1 * f[0] + omega * R(1.0 / 3.0) * K;
    if (FORCED) post0 -= (R(1) - R(0.5) * omega) * vb;  // w_0 (1 - omega/2) (-3 v.b), w_0 = 1/3
    put(out(0, c), post0);
#pragma unroll
    for (int q = 0; q < NP; q++) {
        const int i = 2 * q + 1;
        const bool face = i < 7;
        R eu = 0, eb = 0;
        if (cx(i) > 0) eu += vx;
        if (cx(i) < 0) eu -= vx;
        if (cy(i) > 0) eu += vy;
        if (cy(i) < 0) eu -= vy;
        if (cz(i) > 0) eu += vz;
        if (cz(i) < 0) eu -= vz;
        R A = (face ? a1 : a2) * eu * eu + (face ? wK1 : wK2);
        R B = (face ? b1 : b2) * eu;
        if (FORCED) {
            if (cx(i) > 0) eb += bx;
            if (cx(i) < 0) eb -= bx;
            if (cy(i) > 0) eb += by;
            if (cy(i) < 0) eb -= by;
            if (cz(i) > 0) eb += bz;
            if (cz(i) < 0) eb -= bz;
            const R kw = face ? kw1 : kw2;
            A += kw * (R(9) * eu * eb - R(3) * vb);
            B += R(3) * kw * eb;
        }
        put(out(i, c), om1 * f[i] + (A + B));
        put(out(i + 1, c), om1 * f[i + 1] + (A - B));
    }
    return Moments<R>{sd, jx, jy, jz};
}

}  // namespace lbm

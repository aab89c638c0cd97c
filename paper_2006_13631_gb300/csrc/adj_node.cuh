// Arithmetic of the adjoint at one node: derivatives of the equilibrium, of the
// states that the interpolations carry, and of a patch node's FV update.
//
// Reverse mode of one lattice step, with every decision of the forward step
// held fixed (node classes, refill types, donor cells and triangles: the map
// is smooth in the states and parameters between decisions).  Adjoints have the
// population type; a parameter's sum takes every product in FP64.  Notation: for a deviation set f (f_i = f'_i), rho = rho0 + dr,
// u = j / rho; the equilibrium's derivatives are
//   d feq_i / d dr |_u = A_i = w_i (1 + 3 c.u + 4.5 (c.u)^2 - 1.5 u^2),
//   d feq_i / d u      = B_i = w_i rho (3 c_i + 9 (c.u) c_i - 3 u),
// so that d feq_i / d f_j = A_i + B_i . (c_j - u) / rho, and the transpose
// product is (J^T l)_j = a + b . (c_j - u) / rho with a = sum_i l_i A_i,
// b = sum_i l_i B_i.
// The sums run over pairs of opposite directions (c_opp = -c_i: the even terms
// take l_i + l_opp, the odd ones l_i - l_opp) and use 1 / rho once: an FP64
// division is some ten FP64 instructions, which issue at 1/64 of the FP32 rate.
#pragma once
#include "fv_node.cuh"

namespace hk {

template <typename R>
__device__ __forceinline__ void mom_d(const R (&f)[9], R rho0, R& dr, R& rho, R& ux, R& uy, R& inv) {
    R m0, mx, my;
    pops_moments(pops_of(f), m0, mx, my);
    dr = m0;
    rho = rho0 + m0;
    inv = R(1) / rho;
    ux = mx * inv;
    uy = my * inv;
}
template <typename R>
__device__ __forceinline__ void mom_d(const R (&f)[9], R rho0, R& dr, R& rho, R& ux, R& uy) {
    R inv;
    mom_d(f, rho0, dr, rho, ux, uy, inv);
}

// f_i^eq - w_i rho0 for all i
template <typename R>
__device__ __forceinline__ void feq_all(R dr, R rho, R ux, R uy, R (&e)[9]) {
    const R q = R(-1.5) * (ux * ux + uy * uy);
    e[0] = w_of<R>(0) * (dr + rho * q);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        if (opp_of(i) < i) continue;
        const R cu = cdot(i, ux, uy), G = dr + rho * (R(4.5) * cu * cu + q), H = rho * (R(3) * cu);
        e[i] = w_of<R>(i) * (G + H);
        e[opp_of(i)] = w_of<R>(i) * (G - H);
    }
}

// a = sum_i l_i A_i, b = sum_i l_i B_i / rho at velocity u
template <typename R>
__device__ __forceinline__ void feq_ab(R ux, R uy, const R (&l)[9], R& a, R& bx, R& by) {
    const R z = R(1) - R(1.5) * (ux * ux + uy * uy);
    R ws = w_of<R>(0) * l[0];
    a = z * ws;
    R tx = R(0), ty = R(0);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        if (opp_of(i) < i) continue;
        const R s = l[i] + l[opp_of(i)], d = l[i] - l[opp_of(i)], cu = cdot(i, ux, uy), w = w_of<R>(i);
        a += w * ((z + R(4.5) * cu * cu) * s + R(3) * cu * d);
        const R t = w * (R(3) * d + R(9) * cu * s);
        ws += w * s;
        tx = add_cx(i, tx, t);
        ty = add_cy(i, ty, t);
    }
    bx = tx - R(3) * ux * ws;
    by = ty - R(3) * uy * ws;
}

// out += scale * (g + b . c_j)
template <typename R>
__device__ __forceinline__ void lin_add(R g, R bx, R by, R scale, R (&out)[9]) {
    out[0] += scale * g;
#pragma unroll
    for (int j = 1; j < 9; ++j) out[j] += scale * (g + cdot(j, bx, by));
}

// out += scale * J_feq(f)^T lam, J at the velocity u of f
template <typename R>
__device__ __forceinline__ void jfeqT_add(R ux, R uy, const R (&lam)[9], R scale, R (&out)[9]) {
    R a, bx, by;
    feq_ab(ux, uy, lam, a, bx, by);
    lin_add(a - bx * ux - by * uy, bx, by, scale, out);
}

// the interpolated state s(f) = (dr, ux, uy, f^neq[9]) of a deviation set
template <typename R>
__device__ __forceinline__ void state_d(const R (&f)[9], R rho0, R (&st)[12]) {
    R dr, rho, ux, uy, e[9];
    mom_d(f, rho0, dr, rho, ux, uy);
    st[0] = dr;
    st[1] = ux;
    st[2] = uy;
    feq_all(dr, rho, ux, uy, e);
#pragma unroll
    for (int i = 0; i < 9; ++i) st[3 + i] = f[i] - e[i];
}

// out += scale * (d s / d f)^T ls, st the state of the set
template <typename R>
__device__ __forceinline__ void stateT_add(const R (&st)[12], R rho0, const R (&ls)[12], R scale, R (&out)[9]) {
    const R inv = R(1) / (rho0 + st[0]), ux = st[1], uy = st[2];
    R ln[9], a, bx, by;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        ln[j] = ls[3 + j];
        out[j] += scale * ls[3 + j];
    }
    feq_ab(ux, uy, ln, a, bx, by);
    const R gx = ls[1] * inv - bx, gy = ls[2] * inv - by;
    lin_add(ls[0] - a - gx * ux - gy * uy, gx, gy, scale, out);
}

// f = f^eq(st) + k f^neq(st) (eq. continuity_stresses with k = 1 - 1/(2 tau_s),
// eq. postcollision2_s with k = 2 (tau_s - 1)/(2 tau_s - 1)): ls = (d f / d st)^T lf,
// lk += d f / d k . lf
template <typename R>
__device__ __forceinline__ void ffsT(const R (&st)[12], R rho0, R k, const R (&lf)[9], R (&ls)[12], double& lk) {
    const R rho = rho0 + st[0];
    R a, bx, by;
    feq_ab(st[1], st[2], lf, a, bx, by);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        ls[3 + i] = k * lf[i];
        lk += double(lf[i] * st[3 + i]);
    }
    ls[0] = a;
    ls[1] = rho * bx;
    ls[2] = rho * by;
}

// ---- a quad's share of the reverse FV sub-step (k_adj_fv_rev): lane q holds the
// pair of opposite directions q, lane 0 also f0
template <typename T>
struct AQuad {
    int q, ia, ib;
    T w;    // weight of the lane's directions
    T sgn;  // +1 where the first direction's c . g is +g (lanes 0 .. 2), -1 on lane 3
};
template <typename T>
__device__ __forceinline__ AQuad<T> aquad() {
    AQuad<T> Q;
    Q.q = threadIdx.x & 3;
    Q.ia = Q.q < 2 ? Q.q : Q.q + 2;
    Q.ib = Q.ia + 2;
    Q.w = w_of<T>(Q.q < 2 ? 1 : 5);
    Q.sgn = Q.q == 3 ? T(-1) : T(1);
    return Q;
}
template <typename T>
__device__ __forceinline__ T aq_shfl(T v, int src) {
    return __shfl_sync(0xffffffffu, v, src, 4);
}
template <typename T>
__device__ __forceinline__ T aq_sum(T v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
template <typename T>
__device__ __forceinline__ T aq_dot(const AQuad<T>& Q, T x, T y) {
    return Q.q == 0 ? x : Q.q == 1 ? y : Q.sgn * x + y;
}
// a = sum_i l_i A_i and b = sum_i l_i B_i / rho at velocity u of the set l
// (pair la, lb on each lane, l0 on lane 0): see feq_ab
template <typename T>
__device__ __forceinline__ void aq_feq(const AQuad<T>& Q, T ux, T uy, T la, T lb, T l0, T& a, T& bx, T& by) {
    const T s = la + lb, dd = la - lb, cu = aq_dot(Q, ux, uy), us = T(1) - T(1.5) * (ux * ux + uy * uy);
    const T z = Q.q == 0 ? w_of<T>(0) * l0 : T(0);
    const T ws = aq_sum(Q.w * s + z);
    a = aq_sum(Q.w * ((us + T(4.5) * cu * cu) * s + T(3) * cu * dd) + us * z);
    const T t = Q.w * (T(3) * dd + T(9) * cu * s);
    const T t2 = aq_shfl(t, 2), t3 = aq_shfl(t, 3);
    bx = aq_shfl(t, 0) + (t2 - t3) - T(3) * ux * ws;
    by = aq_shfl(t, 1) + (t2 + t3) - T(3) * uy * ws;
}

// What a quad holds of its node: at outer nodes the lattice state at t and
// t + 1 (drho, ux, uy, f^neq of the lane's pair and f^neq_0) and the sums of
// its adjoint (the lane's share: its pair, and f^neq_0 with drho, ux or uy);
// kq: in FP32, the lane's products of the sum of kneq at the latest sub-step
template <typename T>
struct ANode {
    int k;
    int8_t kind;
    bool valid;
    T s0[6], s1[6];
    T g0[4], g1[4];
    T kq[3];
};
// what sub-step m's record gives the lane: its collision sums and the wall moments
template <typename T>
struct ARec {
    T na, nb, n0, rho, wx, wy;
};

// psi at the quad's node for a sub-step (time fraction th, wall velocity U, V,
// record r) from the adjoint (la, lb, l0) of the state after it, the outer
// nodes' feed adjoint, and the parameter terms (1/tau_u, wall velocity, kneq; in
// FP32 that of kneq is left to adj_kneq)
template <typename T>
__device__ __forceinline__ void adj_psi(const Dev<T>& d, const AQuad<T>& Q, ANode<T>& N, const ARec<T>& r, T th, T U, T V,
                                        T la, T lb, T l0, T& pa, T& pb, T& p0, T& l_inv, double& l_kneq, T& l_v) {
    pa = la, pb = lb, p0 = l0;
    const bool wall = N.kind == HLBM_NODE_WALL, outer = N.kind == HLBM_NODE_OUTER;
    if (__any_sync(0xffffffffu, wall)) {
        // g(f) = f + f^eq(rho, U) - f^eq(rho, u(f))
        T a1, bx1, by1, a2, bx2, by2;
        aq_feq(Q, U, V, la, lb, l0, a1, bx1, by1);
        aq_feq(Q, r.wx, r.wy, la, lb, l0, a2, bx2, by2);
        if (wall) {
            const T g = a1 - a2 + bx2 * r.wx + by2 * r.wy, c = aq_dot(Q, bx2, by2);
            pa += g - c;
            pb += g + c;
            p0 += g;
            if (Q.q == 0) l_v += r.rho * by1;
        }
    }
    if (__any_sync(0xffffffffu, outer)) {
        const T t0 = T(1) - th;
        T st[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) st[j] = t0 * N.s0[j] + th * N.s1[j];
        T a, bx, by;
        aq_feq(Q, st[1], st[2], la, lb, l0, a, bx, by);
        if (outer) {
            const T rho = d.rho0 + st[0];
            const T v[4] = {d.kneq * la, d.kneq * lb, d.kneq * l0, Q.q == 0 ? a : rho * (Q.q == 1 ? bx : by)};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                N.g0[j] += t0 * v[j];
                N.g1[j] += th * v[j];
            }
            if constexpr (sizeof(T) == 4) {
                N.kq[0] = la * st[3];
                N.kq[1] = lb * st[4];
                N.kq[2] = Q.q == 0 ? l0 * st[5] : T(0);
            } else {
                l_kneq += la * st[3] + lb * st[4] + (Q.q == 0 ? l0 * st[5] : T(0));
            }
            pa = pb = p0 = T(0);
        }
    }
    if (!N.valid) return;
    l_inv -= d.dt_u * (pa * r.na + pb * r.nb + (Q.q == 0 ? p0 * r.n0 : T(0)));
}
// FP32: the outer node's terms of kneq into the FP64 sum, once psi is on its way.
// (The conversions and FP64 additions within adj_psi: reverse sweep of 160 steps
// of the 2588-node patch, n = 96, 101 ms instead of 94; an FP32 sum of the three
// products: 90.5.)
template <typename T>
__device__ __forceinline__ void adj_kneq(const ANode<T>& N, double& l_kneq) {
    if constexpr (sizeof(T) == 4) {
        if (N.kind != HLBM_NODE_OUTER) return;
#pragma unroll
        for (int j = 0; j < 3; ++j) l_kneq += double(N.kq[j]);
    }
}

}  // namespace hk

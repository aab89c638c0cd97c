// Arithmetic of one patch node's FV update (eq. ulbe), shared by every FV
// kernel.  All operations are explicitly rounded and each result element has
// one expression, so a node's bits depend neither on the kernel nor on how
// the elements are grouped into instructions.
//
// Populations are handled in pairs: A = (f1, f2), B = (f3, f4), C = (f5, f6),
// D = (f7, f8) and E = (f0, z0), F = (z1, z2), z being the quadratic
// equilibrium terms of z_of.  Opposite directions are (A, B) and (C, D)
// element by element, so the moments of a set are sums and differences of
// pairs.  In FP32 a pair lives in one 64-bit register pair and each operation
// is one packed instruction (fma.rn.f32x2 and the like, each half rounded as
// the scalar one): the update of the 4096^2 patch is bound by the instructions
// it issues (issue slots 52 % busy, FP32 pipes far below their peak), and the
// packed form halves those of the row sums and of the collision.  FP64 pairs
// are two scalar operations.
#pragma once
#include "hlbm_dev.cuh"

namespace hk {

template <typename T>
struct Pr;
template <>
struct Pr<float> {
    unsigned long long v;
};
template <>
struct Pr<double> {
    double a, b;
};

__device__ __forceinline__ Pr<float> pk(float a, float b) {
    Pr<float> p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.v) : "f"(a), "f"(b));
    return p;
}
__device__ __forceinline__ Pr<double> pk(double a, double b) { return Pr<double>{a, b}; }
__device__ __forceinline__ float px(Pr<float> p) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
    return a;
}
__device__ __forceinline__ float py(Pr<float> p) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v));
    return b;
}
__device__ __forceinline__ double px(Pr<double> p) { return p.a; }
__device__ __forceinline__ double py(Pr<double> p) { return p.b; }
__device__ __forceinline__ Pr<float> padd(Pr<float> a, Pr<float> b) {
    Pr<float> r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pr<float> psub(Pr<float> a, Pr<float> b) {
    Pr<float> r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pr<float> pmul(Pr<float> a, Pr<float> b) {
    Pr<float> r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Pr<float> pfma(Pr<float> a, Pr<float> b, Pr<float> c) {
    Pr<float> r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ Pr<double> padd(Pr<double> a, Pr<double> b) {
    return Pr<double>{__dadd_rn(a.a, b.a), __dadd_rn(a.b, b.b)};
}
__device__ __forceinline__ Pr<double> psub(Pr<double> a, Pr<double> b) {
    return Pr<double>{__dsub_rn(a.a, b.a), __dsub_rn(a.b, b.b)};
}
__device__ __forceinline__ Pr<double> pmul(Pr<double> a, Pr<double> b) {
    return Pr<double>{__dmul_rn(a.a, b.a), __dmul_rn(a.b, b.b)};
}
__device__ __forceinline__ Pr<double> pfma(Pr<double> a, Pr<double> b, Pr<double> c) {
    return Pr<double>{__fma_rn(a.a, b.a, c.a), __fma_rn(a.b, b.b, c.b)};
}

// the eight moving populations of a set, and its rest population
template <typename T>
struct Pops {
    Pr<T> A, B, C, D;
    T f0;
};

template <typename T>
__device__ __forceinline__ Pops<T> pops_of(const T (&f)[9]) {
    return Pops<T>{pk(f[1], f[2]), pk(f[3], f[4]), pk(f[5], f[6]), pk(f[7], f[8]), f[0]};
}
template <typename T>
__device__ __forceinline__ void pops_to(const Pops<T>& p, T (&f)[9]) {
    f[0] = p.f0;
    f[1] = px(p.A), f[2] = py(p.A), f[3] = px(p.B), f[4] = py(p.B);
    f[5] = px(p.C), f[6] = py(p.C), f[7] = px(p.D), f[8] = py(p.D);
}

// The state (drho, ux, uy, f^neq) that the interpolations between the grids
// carry (Sec. 4, eq. postcollision2_s): pairs of opposite directions share the
// even and odd parts of f^eq, and 1 / rho is formed once.
template <typename T>
__device__ __forceinline__ void state_of(const T (&f)[9], T rho0, T (&st)[12]);

// sum f_i, sum c_ix f_i, sum c_iy f_i
__device__ __forceinline__ void pops_moments(const Pops<float>& p, float& m0, float& mx, float& my) {
    float f[9];
    pops_to(p, f);
    m0 = f[0];
    mx = my = 0.0f;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        m0 = add_rn(m0, f[i]);
        mx = add_cx(i, mx, f[i]);
        my = add_cy(i, my, f[i]);
    }
}
__device__ __forceinline__ void pops_moments(const Pops<double>& p, double& m0, double& mx, double& my) {
    const Pr<double> s1 = padd(p.A, p.B), d1 = psub(p.A, p.B), s2 = padd(p.C, p.D), d2 = psub(p.C, p.D);
    m0 = add_rn(p.f0, add_rn(add_rn(px(s1), py(s1)), add_rn(px(s2), py(s2))));
    mx = add_rn(px(d1), sub_rn(px(d2), py(d2)));
    my = add_rn(py(d1), add_rn(px(d2), py(d2)));
}

// (f_i^eq - w_i rho0) / w_i of the directions with c . u = c (x) and of their
// opposites (y): drho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u^2)
__device__ __forceinline__ void feq_x(Pr<float> c, float dr, float rho, float usq, Pr<float>& x, Pr<float>& y) {
    const Pr<float> e = pmul(pmul(pk(4.5f, 4.5f), c), c), u = pk(usq, usq), m = pk(-1.5f, -1.5f), r = pk(rho, rho), d = pk(dr, dr);
    x = pfma(r, pfma(m, u, pfma(pk(3.0f, 3.0f), c, e)), d);
    y = pfma(r, pfma(m, u, pfma(pk(-3.0f, -3.0f), c, e)), d);
}
// all of them, as a set: the axes' and the diagonals' pairs, and the rest one
__device__ __forceinline__ Pops<float> feq_x(float dr, float rho, float ux, float uy) {
    const float usq = fma_rn(ux, ux, mul_rn(uy, uy));
    Pops<float> X;
    feq_x(pk(ux, uy), dr, rho, usq, X.A, X.B);
    feq_x(pk(add_rn(ux, uy), sub_rn(uy, ux)), dr, rho, usq, X.C, X.D);
    X.f0 = fma_rn(rho, mul_rn(-1.5f, usq), dr);
    return X;
}

// f_i^eq - w_i rho0 of the pair (i, opp(i)) as w_i (G + H), w_i (G - H)
template <typename T>
__device__ __forceinline__ void feq_pair(int i, T dr, T rho, T ux, T uy, T q, T& a, T& b) {
    const T cu = cdot(i, ux, uy);
    const T G = fma_rn(rho, fma_rn(mul_rn(T(4.5), cu), cu, q), dr), H = mul_rn(rho, mul_rn(T(3), cu));
    a = mul_rn(w_of<T>(i), add_rn(G, H));
    b = mul_rn(w_of<T>(i), sub_rn(G, H));
}
template <typename T>
__device__ __forceinline__ void state_of(const T (&f)[9], T rho0, T (&st)[12]) {
    T dr, jx, jy;
    pops_moments(pops_of(f), dr, jx, jy);
    const T rho = add_rn(rho0, dr), inv = T(1) / rho, ux = mul_rn(jx, inv), uy = mul_rn(jy, inv);
    st[0] = dr;
    st[1] = ux;
    st[2] = uy;
    if constexpr (sizeof(T) == 4) {
        T x[9];
        pops_to(feq_x(dr, rho, ux, uy), x);
#pragma unroll
        for (int i = 0; i < 9; ++i) st[3 + i] = fma_rn(-w_of<T>(i), x[i], f[i]);
        return;
    }
    const T q = mul_rn(T(-1.5), fma_rn(ux, ux, mul_rn(uy, uy)));
    st[3] = sub_rn(f[0], mul_rn(w_of<T>(0), fma_rn(rho, q, dr)));
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        if (opp_of(i) < i) continue;
        T a, b;
        feq_pair(i, dr, rho, ux, uy, q, a, b);
        st[3 + i] = sub_rn(f[i], a);
        st[3 + opp_of(i)] = sub_rn(f[opp_of(i)], b);
    }
}

// FP32: acc - w_i (4.5 Q_i + 3 c_i . (x, y) + g) with Q the quadratic part (qa on
// the axes, qd on the diagonals) when kQuad
template <bool kQuad>
__device__ __forceinline__ void pops_sub_lin(Pops<float>& p, float g, float x, float y, Pr<float> qa, Pr<float> qd) {
    const Pr<float> w1 = pk(-w_of<float>(1), -w_of<float>(1)), w5 = pk(-w_of<float>(5), -w_of<float>(5));
    const Pr<float> h = pk(4.5f, 4.5f), t = pk(3.0f, 3.0f), m = pk(-3.0f, -3.0f), gg = pk(g, g);
    const Pr<float> ca = pk(x, y), cd = pk(add_rn(x, y), sub_rn(y, x));
    Pr<float> A = pfma(t, ca, gg), B = pfma(m, ca, gg), C = pfma(t, cd, gg), D = pfma(m, cd, gg);
    if (kQuad) A = pfma(h, qa, A), B = pfma(h, qa, B), C = pfma(h, qd, C), D = pfma(h, qd, D);
    p.A = pfma(w1, A, p.A);
    p.B = pfma(w1, B, p.B);
    p.C = pfma(w5, C, p.C);
    p.D = pfma(w5, D, p.D);
}

// FP64: acc - w_i (G_i + 3 c_i . (x, y)) over the moving directions, G = (g1, g2)
// on the axes x and y and (g5, g6) on the diagonals (1, 1) and (-1, 1)
template <typename T>
__device__ __forceinline__ void pops_sub_lin(Pops<T>& p, Pr<T> ga, Pr<T> gd, T x, T y) {
    const Pr<T> three = pk(T(3), T(3)), w1 = pk(-w_of<T>(1), -w_of<T>(1)), w5 = pk(-w_of<T>(5), -w_of<T>(5));
    const Pr<T> ha = pmul(three, pk(x, y)), hd = pmul(three, pk(add_rn(x, y), sub_rn(y, x)));
    p.A = pfma(w1, padd(ga, ha), p.A);
    p.B = pfma(w1, psub(ga, ha), p.B);
    p.C = pfma(w5, padd(gd, hd), p.C);
    p.D = pfma(w5, psub(gd, hd), p.D);
}

// Patch record: f'[0..8] and the quadratic equilibrium terms
// z = (jx^2 / rho, jx jy / rho, jy^2 / rho) at [9..11].  With j = sum_i c_i f'_i
// and drho = sum_i f'_i,
//   f_i^eq - w_i rho0 = w_i (drho - 1.5 (z0 + z2) + 3 c_i.j + 4.5 (cx^2 z0 + 2 cx cy z1 + cy^2 z2)),
// linear in (drho, j, z).  For sum_k C_Pk f^eq(P_k) the drho and j parts
// are sums of Cf_i = sum_k C_Pk f'_k,i, so only z has to be carried.
template <typename T>
__device__ __forceinline__ void z_of(const Pops<T>& p, T rho0, T (&z)[3], T& ux, T& uy) {
    T dr, jx, jy;
    pops_moments(p, dr, jx, jy);
    const T inv = T(1) / add_rn(rho0, dr);
    ux = mul_rn(jx, inv);
    uy = mul_rn(jy, inv);
    if constexpr (sizeof(T) == 4) {
        z[0] = mul_rn(mul_rn(jx, jx), inv);
        z[1] = mul_rn(mul_rn(jx, jy), inv);
        z[2] = mul_rn(mul_rn(jy, jy), inv);
    } else {
        z[0] = mul_rn(jx, ux);
        z[1] = mul_rn(jx, uy);
        z[2] = mul_rn(jy, uy);
    }
}
template <typename T>
__device__ __forceinline__ void z_of(const T (&f)[9], T rho0, T (&z)[3]) {
    T ux, uy;
    z_of(pops_of(f), rho0, z, ux, uy);
}

// The sums of one row (eq. ulbe), off-diagonal entries in row order, then the
// pivot.  With the exact zero row sum g_PP = -sum_k g_Pk the streaming sums
// are S_i = sum_{k != P} (c_i . g_Pk) (f_k,i - f_P,i): the same number in
// exact arithmetic, but the differences are small next to f_k, so that in
// FP32 the products do not round at the scale of |g| |f| (|g| ~ 1/h, h down
// to 0.1 at the wall).  S is accumulated with the positive one of each pair
// of opposite coefficients: gx, gy on the axes, gx + gy and gx - gy on the
// diagonals (S_3, S_4, S_6, S_7 change sign at the end).
template <typename T>
struct FvSums {
    Pr<T> SA, SB, SC, SD;  // streaming sums
    Pr<T> A, B, C, D, E, F;  // sum_k C_Pk of the record's pairs
};

template <typename T>
__device__ __forceinline__ void fv_sums_init(FvSums<T>& s) {
    const Pr<T> o = pk(T(0), T(0));
    s.SA = s.SB = s.SC = s.SD = s.A = s.B = s.C = s.D = s.E = s.F = o;
}

// a record's pairs
template <typename T>
struct RecP {
    Pr<T> A, B, C, D, E, F;
};

template <typename T>
__device__ __forceinline__ void fv_sums_entry(FvSums<T>& s, T gx, T gy, T c, const RecP<T>& f, const Pops<T>& P) {
    const Pr<T> ga = pk(gx, gy), gd = pk(add_rn(gx, gy), sub_rn(gx, gy)), cc = pk(c, c);
    s.SA = pfma(ga, psub(f.A, P.A), s.SA);
    s.SB = pfma(ga, psub(f.B, P.B), s.SB);
    s.SC = pfma(gd, psub(f.C, P.C), s.SC);
    s.SD = pfma(gd, psub(f.D, P.D), s.SD);
    s.A = pfma(cc, f.A, s.A);
    s.B = pfma(cc, f.B, s.B);
    s.C = pfma(cc, f.C, s.C);
    s.D = pfma(cc, f.D, s.D);
    s.E = pfma(cc, f.E, s.E);
    s.F = pfma(cc, f.F, s.F);
}

// The update of eq. ulbe from the sums, own record P and C_PP.  The collision
// sums Cf_i - ceq_i carry no mass and no momentum in exact arithmetic (ceq is
// built from the moments of Cf); their rounding residues m0 = sum_i n_i,
// m = sum_i c_i n_i are removed by subtracting w_i (m0 + 3 c_i.m), which
// leaves exact values unchanged and stops the residues from acting, sub-step
// after sub-step, as spurious sources of mass and momentum.
// n receives the collision sums (residues removed).
template <typename T>
__device__ __forceinline__ Pops<T> fv_sums_finish(const Dev<T>& d, FvSums<T>& s, T cP, const RecP<T>& P, Pops<T>& n) {
    const Pr<T> cc = pk(cP, cP);
    n.A = pfma(cc, P.A, s.A);
    n.B = pfma(cc, P.B, s.B);
    n.C = pfma(cc, P.C, s.C);
    n.D = pfma(cc, P.D, s.D);
    const Pr<T> e = pfma(cc, P.E, s.E), f = pfma(cc, P.F, s.F);
    n.f0 = px(e);
    const T Z0 = py(e), Z1 = px(f), Z2 = py(f);
    T dr, jx, jy;
    pops_moments(n, dr, jx, jy);
    // sum_k C_Pk (f^eq_k,i - w_i rho0): quadratic part Z0, Z2 on the axes and
    // Z0 + Z2 +- 2 Z1 on the diagonals
    const T zs = add_rn(Z0, Z2), q0 = fma_rn(T(-1.5), zs, dr);
    if constexpr (sizeof(T) == 4) {
        const Pr<T> qd = pk(add_rn(fma_rn(T(2), Z1, Z0), Z2), add_rn(fma_rn(T(-2), Z1, Z0), Z2));
        pops_sub_lin<true>(n, q0, jx, jy, pk(Z0, Z2), qd);
    } else {
        const Pr<T> q = pk(q0, q0), h = pk(T(4.5), T(4.5));
        pops_sub_lin(n, pfma(h, pk(Z0, Z2), q), pfma(h, pk(fma_rn(T(2), Z1, zs), fma_rn(T(-2), Z1, zs)), q), jx, jy);
    }
    n.f0 = fma_rn(-w_of<T>(0), q0, n.f0);
    T m0, mx, my;
    pops_moments(n, m0, mx, my);
    const Pr<T> mm = pk(m0, m0);
    if constexpr (sizeof(T) == 4)
        pops_sub_lin<false>(n, m0, mx, my, mm, mm);
    else
        pops_sub_lin(n, mm, mm, mx, my);
    n.f0 = fma_rn(-w_of<T>(0), m0, n.f0);
    // f_P + dt_u (S - n / tau_u)
    const T iv = d.inv_tau_u, dt = d.dt_u;
    Pops<T> o;
    o.A = pfma(pk(dt, dt), pfma(pk(-iv, -iv), n.A, s.SA), P.A);
    o.B = pfma(pk(-dt, -dt), pfma(pk(iv, iv), n.B, s.SB), P.B);
    o.C = pfma(pk(dt, -dt), pfma(pk(-iv, iv), n.C, s.SC), P.C);
    o.D = pfma(pk(-dt, dt), pfma(pk(iv, -iv), n.D, s.SD), P.D);
    o.f0 = fma_rn(dt, mul_rn(-iv, n.f0), px(P.E));
    return o;
}

// wall nodes: impose the lamina velocity, keep the non-equilibrium part:
// f_i += f_i^eq(rho, U) - f_i^eq(rho, u); in FP64
// w_i rho (3 c_i.(U - u) + 4.5 ((c_i.U)^2 - (c_i.u)^2) - 1.5 (U^2 - u^2)),
// the squares as products of sums and differences
// (the update's moments rho, u go to mo)
template <typename T>
__device__ __forceinline__ void fv_wall(const Dev<T>& d, T U, T V, Pops<T>& p, T (&mo)[3]) {
    T dr, jx, jy;
    pops_moments(p, dr, jx, jy);
    const T rho = add_rn(d.rho0, dr), inv = T(1) / rho;
    const T ux = mul_rn(jx, inv), uy = mul_rn(jy, inv);
    mo[0] = rho;
    mo[1] = ux;
    mo[2] = uy;
    if constexpr (sizeof(T) == 4) {
        const Pops<T> X = feq_x(dr, rho, U, V), Y = feq_x(dr, rho, ux, uy);
        auto add = [](T wi, Pr<T> x, Pr<T> y, Pr<T> f) { return padd(f, pfma(pk(wi, wi), x, pmul(pk(-wi, -wi), y))); };
        p.A = add(w_of<T>(1), X.A, Y.A, p.A);
        p.B = add(w_of<T>(1), X.B, Y.B, p.B);
        p.C = add(w_of<T>(5), X.C, Y.C, p.C);
        p.D = add(w_of<T>(5), X.D, Y.D, p.D);
        p.f0 = add_rn(p.f0, fma_rn(w_of<T>(0), X.f0, mul_rn(-w_of<T>(0), Y.f0)));
        return;
    }
    const T dx = sub_rn(U, ux), dy = sub_rn(V, uy), sx = add_rn(U, ux), sy = add_rn(V, uy);
    const T b = mul_rn(T(-1.5), fma_rn(dx, sx, mul_rn(dy, sy)));
    const Pr<T> bb = pk(b, b), h = pk(T(4.5), T(4.5)), three = pk(T(3), T(3));
    const Pr<T> da = pk(dx, dy), dd = pk(add_rn(dx, dy), sub_rn(dy, dx));
    const Pr<T> ga = pfma(pmul(h, da), pk(sx, sy), bb), gd = pfma(pmul(h, dd), pk(add_rn(sx, sy), sub_rn(sy, sx)), bb);
    const Pr<T> ha = pmul(three, da), hd = pmul(three, dd);
    const T w1 = mul_rn(w_of<T>(1), rho), w5 = mul_rn(w_of<T>(5), rho);
    p.A = pfma(pk(w1, w1), padd(ga, ha), p.A);
    p.B = pfma(pk(w1, w1), psub(ga, ha), p.B);
    p.C = pfma(pk(w5, w5), padd(gd, hd), p.C);
    p.D = pfma(pk(w5, w5), psub(gd, hd), p.D);
    p.f0 = fma_rn(mul_rn(w_of<T>(0), rho), b, p.f0);
}

// outer nodes: the lattice state interpolated linearly in time (eq. 182,
// Dirichlet reading); sn[j * stride], j < 12, is the state (drho, ux, uy,
// f^neq) at t and sn[(12 + j) * stride] the one at t + 1;
// f = f^eq(rho, u) + (1 - 1/(2 tau_s)) f^neq
template <typename T>
__device__ __forceinline__ Pops<T> fv_outer_from(const Dev<T>& d, const T* sn, int64_t stride, int m) {
    const T th = T(m + 1) / T(d.n_sub), t0 = sub_rn(T(1), th);
    auto at = [&](int j) { return fma_rn(t0, sn[j * stride], mul_rn(th, sn[(12 + j) * stride])); };
    const T dr = at(0), ux = at(1), uy = at(2), rho = add_rn(d.rho0, dr);
    if constexpr (sizeof(T) == 4) {
        const Pops<T> X = feq_x(dr, rho, ux, uy);
        auto f = [&](T wi, Pr<T> x, int j) { return pfma(pk(d.kneq, d.kneq), pk(at(j), at(j + 1)), pmul(pk(wi, wi), x)); };
        Pops<T> p;
        p.A = f(w_of<T>(1), X.A, 4);
        p.B = f(w_of<T>(1), X.B, 6);
        p.C = f(w_of<T>(5), X.C, 8);
        p.D = f(w_of<T>(5), X.D, 10);
        p.f0 = fma_rn(d.kneq, at(3), mul_rn(w_of<T>(0), X.f0));
        return p;
    }
    const T q = mul_rn(T(-1.5), fma_rn(ux, ux, mul_rn(uy, uy)));
    const Pr<T> rr = pk(rho, rho), qq = pk(q, q), h = pk(T(4.5), T(4.5)), three = pk(T(3), T(3)), kk = pk(d.kneq, d.kneq);
    const Pr<T> ca = pk(ux, uy), cd = pk(add_rn(ux, uy), sub_rn(uy, ux)), dd = pk(dr, dr);
    const Pr<T> ga = pfma(rr, pfma(pmul(h, ca), ca, qq), dd), gd = pfma(rr, pfma(pmul(h, cd), cd, qq), dd);
    const Pr<T> ha = pmul(rr, pmul(three, ca)), hd = pmul(rr, pmul(three, cd));
    const Pr<T> w1 = pk(w_of<T>(1), w_of<T>(1)), w5 = pk(w_of<T>(5), w_of<T>(5));
    Pops<T> p;
    p.A = pfma(kk, pk(at(4), at(5)), pmul(w1, padd(ga, ha)));
    p.B = pfma(kk, pk(at(6), at(7)), pmul(w1, psub(ga, ha)));
    p.C = pfma(kk, pk(at(8), at(9)), pmul(w5, padd(gd, hd)));
    p.D = pfma(kk, pk(at(10), at(11)), pmul(w5, psub(gd, hd)));
    p.f0 = fma_rn(d.kneq, at(3), mul_rn(w_of<T>(0), fma_rn(rho, q, dr)));
    return p;
}

// ---- the same on arrays, for the kernels that keep records in index order
template <typename T>
struct FvAcc {
    T S[9], Cf[9], Z[3];  // S[0] stays 0 (c_0 = 0); signs as in FvSums
};

template <typename T>
__device__ __forceinline__ void fv_acc_init(FvAcc<T>& a) {
#pragma unroll
    for (int i = 0; i < 9; ++i) a.S[i] = a.Cf[i] = T(0);
#pragma unroll
    for (int j = 0; j < 3; ++j) a.Z[j] = T(0);
}

// entry (g_Pk, C_Pk) of row P with the neighbour's state f, z; fP is the
// pivot's state
template <typename T>
__device__ __forceinline__ void fv_acc_entry(FvAcc<T>& a, T gx, T gy, T c, const T (&f)[9], const T (&z)[3],
                                             const T (&fP)[9]) {
    const T gp = add_rn(gx, gy), gm = sub_rn(gx, gy);
    const T g[9] = {T(0), gx, gy, gx, gy, gp, gm, gp, gm};
#pragma unroll
    for (int i = 1; i < 9; ++i) a.S[i] = fma_rn(g[i], sub_rn(f[i], fP[i]), a.S[i]);
#pragma unroll
    for (int i = 0; i < 9; ++i) a.Cf[i] = fma_rn(c, f[i], a.Cf[i]);
#pragma unroll
    for (int k = 0; k < 3; ++k) a.Z[k] = fma_rn(c, z[k], a.Z[k]);
}

template <typename T>
__device__ __forceinline__ void fv_acc_finish(const Dev<T>& d, FvAcc<T>& a, T cP, const T (&fP)[9], const T (&zP)[3],
                                              T (&fn)[9]) {
    FvSums<T> s;
    s.SA = pk(a.S[1], a.S[2]), s.SB = pk(a.S[3], a.S[4]), s.SC = pk(a.S[5], a.S[6]), s.SD = pk(a.S[7], a.S[8]);
    s.A = pk(a.Cf[1], a.Cf[2]), s.B = pk(a.Cf[3], a.Cf[4]), s.C = pk(a.Cf[5], a.Cf[6]), s.D = pk(a.Cf[7], a.Cf[8]);
    s.E = pk(a.Cf[0], a.Z[0]), s.F = pk(a.Z[1], a.Z[2]);
    RecP<T> P;
    P.A = pk(fP[1], fP[2]), P.B = pk(fP[3], fP[4]), P.C = pk(fP[5], fP[6]), P.D = pk(fP[7], fP[8]);
    P.E = pk(fP[0], zP[0]), P.F = pk(zP[1], zP[2]);
    Pops<T> n;
    pops_to(fv_sums_finish(d, s, cP, P, n), fn);
}

template <typename T>
__device__ __forceinline__ void fv_wall(const Dev<T>& d, T U, T V, T (&fn)[9]) {
    Pops<T> p = pops_of(fn);
    T mo[3];
    fv_wall(d, U, V, p, mo);
    pops_to(p, fn);
}

template <typename T>
__device__ __forceinline__ void fv_outer_from(const Dev<T>& d, const T* sn, int64_t stride, int m, T (&fn)[9]) {
    pops_to(fv_outer_from(d, sn, stride, m), fn);
}

}  // namespace hk

// Per-node arithmetic of the two-component Shan-Chen step (paper Sec. 2.1),
// shared by every kernel so that all launch shapes give bit-identical results.
//
// For one node with pulled populations f_is (post-streaming, pre-collision):
//   rho_s = sum_i f_is,  j_s = sum_i f_is c_i                      (Sec. 2.1 moments)
//   g_s = F_s / rho_s = -G sum_i w_i rho_s'(x + c_i) c_i           (Eq. FORCE)
//         [+ A sin(2 pi y / ny) e_x: Kolmogorov forcing, Eq. kolmo]
//   u' = (j_A / tau_A + j_B / tau_B) / (rho_A / tau_A + rho_B / tau_B)
//   f_is += (1 / tau_s) (f^eq_i(rho_s, u' + tau_s g_s) - f_is)      (Eq. eq:be)
// with f^eq_i(rho, u) = w_i rho [1 + 3 c.u + 9/2 (c.u)^2 - 3/2 u.u].
//
// All operations go through Ar<C> (explicitly rounded intrinsics) in a fixed
// order.  The force is taken per unit density, so a vanishing rho_s is never
// divided by.  Momentum and force are summed over opposite-direction pairs
// (the GPU velocity order keeps c_{i+1} = -c_i for odd i): the pair difference
// f_i - f_{i+1}, resp. rho(x + c_i) - rho(x - c_i), is formed first, so both
// vanish exactly in a uniform region and their rounding is antisymmetric.
// Accumulating single terms instead (rho(x + c_i) with an FMA, then
// rho(x - c_i)) leaves a force of about one ulp in uniform regions; in FP32
// that random-walks the total momentum and lets a drop drift by about 1e-5
// lattice units per 1000 steps.  The rest population of the equilibrium is closed as
// f^eq_0 = rho - sum_{i>0} f^eq_i (equal to w_0 rho (...) in exact arithmetic;
// the rounded weights float(1/9), float(4/9), float(1/36) all err upwards and
// would otherwise create about 7e-9 of mass per step at tau = 1), and that
// closure is evaluated as f^eq_0 - f_0 = -sum_{i>0} (f^eq_i - f_i), with
// rho = sum_i f_i: the rest population relaxes by minus the sum of the very
// increments the moving ones receive, so the collision conserves mass up to
// the roundings of that short sum of non-equilibrium parts (a few ulp of
// |f^eq - f|, not of rho) and of the final updates.  Summing rho and
// sum_{i>0} f^eq_i separately instead rounds both at the scale of rho; at
// nodes that repeat the same values those roundings do not average out, and a
// 20000-step FP32 drop drifts in mass by several 1e-6.
#pragma once

#include "sc_common.cuh"

namespace lbmsc {

// rho_s = (f_1 + f_2 + ... + f_{Q-1}) + f_0 of both species, the moving
// populations first and the rest population last, in one fixed order.  rho enters
// the equilibria and the velocity; the closure of f^eq_0 below does not round
// through it.
template <class L, class C> __device__ __forceinline__ Two<C> node_densities(const C (&f)[2][L::Q]) {
    Two<C> r{f[0][1], f[1][1]};
#pragma unroll
    for (int i = 2; i < L::Q; ++i) r = Ar2<C>::add(r, Two<C>{f[0][i], f[1][i]});
    return Ar2<C>::add(r, Two<C>{f[0][0], f[1][0]});
}

template <class L> __host__ __device__ constexpr bool opposite_pairs() {
    for (int i = 1; i + 1 < L::Q; i += 2)
        for (int d = 0; d < 3; ++d)
            if (L::c(i + 1, d) != -L::c(i, d)) return false;
    return L::Q % 2 == 1;
}

// Signed sums of terms in a fixed order.  The first term is taken as it is
// (or negated) rather than added to zero: 0 + x = x for every x but -0, so
// the values are those of the plain running sum, without its first add.
template <class C> struct SignedSum {
    C v;
    bool empty = true;
    __device__ __forceinline__ void add(C x) {
        v = empty ? x : Ar<C>::add(v, x);
        empty = false;
    }
    __device__ __forceinline__ void sub(C x) {
        v = empty ? -x : Ar<C>::sub(v, x);
        empty = false;
    }
    __device__ __forceinline__ C get() const { return empty ? (C)0 : v; }
};

// The same for a Two or an FP64 value (Vops).
template <class V> struct SignedSumV {
    V v;
    bool empty = true;
    __device__ __forceinline__ void add(V x) {
        v = empty ? x : Vops<V>::add(v, x);
        empty = false;
    }
    __device__ __forceinline__ void sub(V x) {
        v = empty ? neg2(x) : Vops<V>::sub(v, x);
        empty = false;
    }
    __device__ __forceinline__ V get() const {
        if (!empty) return v;
        return Vops<V>::c(0);
    }
};

// Momentum of one species, and of both.
template <class L, class C> __device__ __forceinline__ void node_momentum(const C (&f)[L::Q], C (&j)[3]) {
    static_assert(opposite_pairs<L>(), "velocity order must pair c_{i+1} = -c_i");
    SignedSum<C> acc[3];
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const C dlt = Ar<C>::sub(f[i], f[i + 1]);
#pragma unroll
        for (int d = 0; d < L::D; ++d) {
            if (L::c(i, d) == 1) acc[d].add(dlt);
            if (L::c(i, d) == -1) acc[d].sub(dlt);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) j[d] = acc[d].get();
}

template <class L, class C> __device__ __forceinline__ void node_momenta(const C (&f)[2][L::Q], Two<C> (&j)[3]) {
    static_assert(opposite_pairs<L>(), "velocity order must pair c_{i+1} = -c_i");
    SignedSumV<Two<C>> acc[3];
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const Two<C> dlt = Ar2<C>::sub(Two<C>{f[0][i], f[1][i]}, Two<C>{f[0][i + 1], f[1][i + 1]});
#pragma unroll
        for (int d = 0; d < L::D; ++d) {
            if (L::c(i, d) == 1) acc[d].add(dlt);
            if (L::c(i, d) == -1) acc[d].sub(dlt);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) j[d] = acc[d].get();
}

// g_s = -G sum_i w_i rho_s'(x + c_i) c_i for both species; nbr(i) returns the
// pair (rho_A, rho_B) at x + c_i.
template <class L, class C, class Nbr>
__device__ __forceinline__ void node_force(const Nbr& nbr, C G, C (&gA)[3], C (&gB)[3]) {
    using A2 = Ar2<C>;
    static_assert(opposite_pairs<L>(), "velocity order must pair c_{i+1} = -c_i");
    Two<C> g[3] = {both((C)0), both((C)0), both((C)0)};  // (g_B, g_A) / -G: each species feels the other's density
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const C w = (C)L::w(i);
        const Two<C> dr = A2::sub(nbr(i), nbr(i + 1));  // rho(x + c_i) - rho(x - c_i)
#pragma unroll
        for (int d = 0; d < L::D; ++d) {
            if (L::c(i, d) == 1) g[d] = A2::fma(both(w), dr, g[d]);
            if (L::c(i, d) == -1) g[d] = A2::fma(both(-w), dr, g[d]);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const Two<C> h = A2::mul_split(g[d], both(-G));
        gA[d] = h.b;
        gB[d] = h.a;
    }
}

// sin(2 pi y / ny) of the Kolmogorov forcing, y in [0, ny).
template <class C> __device__ __forceinline__ C kolmogorov_sine(int y, int ny);
template <> __device__ __forceinline__ float kolmogorov_sine<float>(int y, int ny) {
    return sinpif(__fdiv_rn((float)(2 * y), (float)ny));
}
template <> __device__ __forceinline__ double kolmogorov_sine<double>(int y, int ny) {
    return sinpi(__ddiv_rn((double)(2 * y), (double)ny));
}

// The Kolmogorov body force of Eq. kolmo (Sec. 4.2), F_x = rho A sin(2 pi y / ny),
// shared by the species in proportion to their densities (F_s,x = rho_s A sin):
// per unit density both g_A and g_B gain b = A sin(2 pi y / ny) along x, which
// then enters the shifted velocities u' + tau_s g_s and the F/2 shift of u_phys.
// A = 0 leaves g untouched.  b depends on the row only, so a kernel whose
// threads keep their row may form it once (kolmogorov_accel) and add it per
// node (node_add_body); node_body_force does both.
template <class C> __device__ __forceinline__ C kolmogorov_accel(C A, int y, int ny) {
    return A == (C)0 ? (C)0 : Ar<C>::mul(A, kolmogorov_sine<C>(y, ny));
}
template <class C> __device__ __forceinline__ void node_add_body(C A, C b, C (&gA)[3], C (&gB)[3]) {
    if (A == (C)0) return;
    gA[0] = Ar<C>::add(gA[0], b);
    gB[0] = Ar<C>::add(gB[0], b);
}
template <class C>
__device__ __forceinline__ void node_body_force(C A, int y, int ny, C (&gA)[3], C (&gB)[3]) {
    if (A == (C)0) return;
    node_add_body<C>(A, kolmogorov_accel<C>(A, y, ny), gA, gB);
}

// c_i . u as a signed sum of u's components (in the order of d).
template <class L, class C> __device__ __forceinline__ C node_cu(int i, const C (&u)[3]) {
    SignedSum<C> cu;
#pragma unroll
    for (int d = 0; d < L::D; ++d) {
        if (L::c(i, d) == 1) cu.add(u[d]);
        if (L::c(i, d) == -1) cu.sub(u[d]);
    }
    return cu.get();
}

template <class L, class V> __device__ __forceinline__ V node_cu2(int i, const V (&u)[3]) {
    SignedSumV<V> cu;
#pragma unroll
    for (int d = 0; d < L::D; ++d) {
        if (L::c(i, d) == 1) cu.add(u[d]);
        if (L::c(i, d) == -1) cu.sub(u[d]);
    }
    return cu.get();
}

// a.b of two vectors, summed from the last component down.
template <class L, class V> __device__ __forceinline__ V node_dot2(const V (&a)[3], const V (&b)[3]) {
    using A = Vops<V>;
    return L::D == 3 ? A::fma(a[0], b[0], A::fma(a[1], b[1], A::mul(a[2], b[2]))) : A::fma(a[0], b[0], A::mul(a[1], b[1]));
}

// The populations the relaxation works on: both species of a node, or one.
template <class L, class C> struct BothF {
    using V = Two<C>;
    C (&f)[2][L::Q];
    __device__ __forceinline__ V get(int i) const { return V{f[0][i], f[1][i]}; }
    __device__ __forceinline__ void set(int i, V v) const {
        f[0][i] = v.a;
        f[1][i] = v.b;
    }
};
template <class L, class C> struct OneF {
    using V = C;
    C (&f)[L::Q];
    __device__ __forceinline__ V get(int i) const { return f[i]; }
    __device__ __forceinline__ void set(int i, V v) const { f[i] = v; }
};

// BGK relaxation towards f^eq(rho_s, u_s), each moving population relaxed as
// soon as its equilibrium is formed (fewer live values), the rest population
// last from the closure f^eq_0 = rho - sum_{i>0} f^eq_i, taken as
// f^eq_0 - f_0 = -sum_{i>0} (f^eq_i - f_i).
template <class L, class F, class V = typename F::V>
__device__ __forceinline__ void node_relax(const F& f, V rho, const V (&u)[3], V omega) {
    using A = Vops<V>;
    const V base = A::fma(A::c(-1.5), node_dot2<L, V>(u, u), A::c(1));
    SignedSumV<V> neq;  // sum_{i>0} (f^eq_i - f_i)
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        const V cu = node_cu2<L, V>(i, u);
        const V wr = A::mul(A::c(L::w(i)), rho);
        const V feq = A::mul_split(wr, A::fma(cu, A::fma(A::c(4.5), cu, A::c(3)), base));
        const V d = A::sub(feq, f.get(i));
        neq.add(d);
        f.set(i, A::fma(omega, d, f.get(i)));
    }
    f.set(0, A::fma(omega, neg2(neq.get()), f.get(0)));
}

// Component s of a pair of vectors.
template <class C> __device__ __forceinline__ void node_part(const Two<C> (&v)[3], int s, C (&o)[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) o[d] = s == 0 ? v[d].a : v[d].b;
}

// Collision of both species of one node: common velocity shifted by tau_s g_s.
// PACK: both species relax together in the packed FP32 instructions, which
// halves the arithmetic instructions of a step (a TMA-fed step is bound by
// issue and by its per-plane barrier as much as by HBM; measured with the
// direct ghost images of store_node: 512^3 FP32 7.66 -> 7.13 ms, 256^3 1.05 ->
// 0.975, Guo forcing at 128^3 0.207 -> 0.180).  The kernels that hold two CTAs
// of 256 threads per SM have 128 registers a thread: the pairs (and their
// constants) then spill, so they relax one species after the other and keep
// only the sums packed (512^3 bf16 rest-offset 5.52 ms packed with 84 bytes of
// spills, 5.28 so, 5.46 before).
template <class L, class C, bool PACK = sizeof(C) == 4>
__device__ __forceinline__ void node_collide(C (&f)[2][L::Q], C rA, C rB, const C (&gA)[3], const C (&gB)[3],
                                             C omega_A, C omega_B, C tau_A, C tau_B) {
    using A = Ar<C>;
    Two<C> j[3], u[3];
    node_momenta<L, C>(f, j);
    const C inv_den = A::rcp(A::fma(rA, omega_A, A::mul(rB, omega_B)));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const C up = A::mul(A::fma(j[d].a, omega_A, A::mul(j[d].b, omega_B)), inv_den);
        u[d] = Ar2<C>::fma(Two<C>{tau_A, tau_B}, Two<C>{gA[d], gB[d]}, both(up));
    }
    if constexpr (PACK) {
        node_relax<L>(BothF<L, C>{f}, Two<C>{rA, rB}, u, Two<C>{omega_A, omega_B});
    } else {
        C us[3];
        node_part<C>(u, 0, us);
        node_relax<L>(OneF<L, C>{f[0]}, rA, us, omega_A);
        node_part<C>(u, 1, us);
        node_relax<L>(OneF<L, C>{f[1]}, rB, us, omega_B);
    }
}

// Guo forcing, the discrete-forcing cure that Sec. 2.3 names for the
// tau-dependent coupling of the velocity shift (the paper prints no formulas;
// this is the standard form, per species, with F_s = rho_s g_s):
//   u_G = sum_s (j_s + F_s / 2) / tau_s / sum_s rho_s / tau_s
//   f_is += (1 / tau_s) (f^eq_i(rho_s, u_G) - f_is) + (1 - 1 / (2 tau_s)) S_is
//   S_is = w_i [3 (c_i - u_G).F_s + 9 (c_i.u_G) (c_i.F_s)]
// The source's rest component is closed as S_0 = -sum_{i>0} S_i (its sum over
// i vanishes in exact arithmetic), and f^eq_0 as in node_relax.  Opposite directions share
// their terms: with t1 = 9 (c.u)(c.F) - 3 u.F and t2 = 3 c.F (c = c_i),
// S_i = w_i (t1 + t2) and S_{i+1} = w_i (t1 - t2), since c_{i+1} = -c_i.
template <class L, class F, class V = typename F::V>
__device__ __forceinline__ void node_relax_guo(const F& f, V rho, const V (&u)[3], const V (&force)[3], V omega) {
    using A = Vops<V>;
    const V base = A::fma(A::c(-1.5), node_dot2<L, V>(u, u), A::c(1));
    const V keep = A::fma(A::c(-0.5), omega, A::c(1));  // 1 - 1 / (2 tau)
    const V m3uF = A::mul(A::c(-3), node_dot2<L, V>(u, force));
    static_assert(opposite_pairs<L>(), "velocity order must pair c_{i+1} = -c_i");
    SignedSumV<V> neq, sources;
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const V cu = node_cu2<L, V>(i, u);  // c_{i+1}.u = -cu exactly (a signed sum of the same terms)
        const V cF = node_cu2<L, V>(i, force);
        const V w = A::c(L::w(i)), ncu = neg2(cu);
        const V wr = A::mul(w, rho);
        const V feq_p = A::mul_split(wr, A::fma(cu, A::fma(A::c(4.5), cu, A::c(3)), base));
        const V feq_m = A::mul_split(wr, A::fma(ncu, A::fma(A::c(4.5), ncu, A::c(3)), base));
        const V d_p = A::sub(feq_p, f.get(i));
        const V d_m = A::sub(feq_m, f.get(i + 1));
        neq.add(d_p);
        neq.add(d_m);
        const V t1 = A::fma(A::mul(A::c(9), cu), cF, m3uF);
        const V t2 = A::mul_split(A::c(3), cF);
        const V src_p = A::mul_split(w, A::add(t1, t2));
        const V src_m = A::mul_split(w, A::sub(t1, t2));
        sources.add(src_p);
        sources.add(src_m);
        f.set(i, A::fma(keep, src_p, A::fma(omega, d_p, f.get(i))));
        f.set(i + 1, A::fma(keep, src_m, A::fma(omega, d_m, f.get(i + 1))));
    }
    f.set(0, A::fma(keep, neg2(sources.get()), A::fma(omega, neg2(neq.get()), f.get(0))));
}

template <class L, class C>
__device__ __forceinline__ void node_collide_guo(C (&f)[2][L::Q], C rA, C rB, const C (&gA)[3], const C (&gB)[3],
                                                 C omega_A, C omega_B) {
    using A = Ar<C>;
    const Two<C> rho{rA, rB};
    Two<C> j[3], F[3], u[3];
    node_momenta<L, C>(f, j);
    const C inv_den = A::rcp(A::fma(rA, omega_A, A::mul(rB, omega_B)));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // rounded before c.F of the diagonal directions adds its components (Ar2: mul_split)
        F[d] = Ar2<C>::mul_split(rho, Two<C>{gA[d], gB[d]});
        const Two<C> m = Ar2<C>::fma(both((C)0.5), F[d], j[d]);
        u[d] = both(A::mul(A::fma(m.a, omega_A, A::mul(m.b, omega_B)), inv_den));
    }
    if constexpr (sizeof(C) == 4) {
        node_relax_guo<L>(BothF<L, C>{f}, rho, u, F, Two<C>{omega_A, omega_B});
    } else {
        C us[3], Fs[3];
        node_part<C>(u, 0, us);
        node_part<C>(F, 0, Fs);
        node_relax_guo<L>(OneF<L, C>{f[0]}, rA, us, Fs, omega_A);
        node_part<C>(F, 1, Fs);
        node_relax_guo<L>(OneF<L, C>{f[1]}, rB, us, Fs, omega_B);
    }
}

// ---- Free-energy (FE) two-population model (Sec. 2.2) ----------------------
// The storage's two "species" hold f_i (density and momentum) and g_i (order
// parameter): rho = sum_i f_i, phi = sum_i g_i, u = sum_i f_i c_i / rho.  The
// free energy is the Eq. FEtau functional with coupling g and gradient
// coefficient kappa; its derivatives come from the isotropic lattice stencils
//   grad phi = 3 sum_i w_i c_i phi(x + c_i),  lap phi = 6 sum_i w_i (phi(x + c_i) - phi(x)),
// formed over opposite pairs like the SC force.  nbr(i).b = phi(x + c_i).
template <class L, class C, class Nbr>
__device__ __forceinline__ void node_fe_derivs(const Nbr& nbr, C phi0, C (&gp)[3], C& lp) {
    using A = Ar<C>;
    static_assert(opposite_pairs<L>(), "velocity order must pair c_{i+1} = -c_i");
    gp[0] = gp[1] = gp[2] = (C)0;
    C lap = (C)0;
    const C two_phi = A::add(phi0, phi0);
#pragma unroll
    for (int i = 1; i < L::Q; i += 2) {
        const C w = (C)L::w(i);
        const C p = nbr(i).b, m = nbr(i + 1).b;
        const C d = A::sub(p, m);  // phi(x + c_i) - phi(x - c_i)
#pragma unroll
        for (int k = 0; k < L::D; ++k) {
            if (L::c(i, k) == 1) gp[k] = A::fma(w, d, gp[k]);
            if (L::c(i, k) == -1) gp[k] = A::fma(-w, d, gp[k]);
        }
        lap = A::fma(w, A::sub(A::add(p, m), two_phi), lap);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) gp[k] = A::mul((C)3, gp[k]);
    lp = A::mul((C)6, lap);
}

// ln x for the chemical potential (the library's log, FP32 or FP64).
__device__ __forceinline__ float fe_log(float x) { return logf(x); }
__device__ __forceinline__ double fe_log(double x) { return log(x); }

// The FE collision of one node (Eqs. FE1, FE2) with the second-order Hermite
// equilibria that meet Eqs. EQFE1 and EQFE2:
//   mu  = cs2/2 ln((rho + phi)/(rho - phi)) - g cs2 phi/2 - kappa lap phi
//   p_b = cs2 rho + g cs2 (rho^2 - phi^2)/4,  s = p_b - kappa phi lap - kappa/2 |grad|^2 - cs2 rho
//   f_i^eq = w_i [rho + 3 rho c.u + 9/2 (s (c.c - D cs2) + kappa ((c.grad)^2 - cs2 |grad|^2)
//                 + rho ((c.u)^2 - cs2 u.u))]
//   g_i^eq = w_i [phi + 3 phi c.u + 9/2 ((Gamma mu - cs2 phi)(c.c - D cs2) + phi ((c.u)^2 - cs2 u.u))]
// (the Hermite term (c_a c_b - cs2 d_ab) M_ab / (2 cs2^2) written out for the
// isotropic-plus-dyadic M of each population), rest components closed as
// rho - sum_{i>0} and phi - sum_{i>0} (each taken, as in node_relax, as minus
// the sum of the moving populations' increments f^eq_i - f_i).  omega = 1/tau, omega_g = 1/tau_g.
template <class L, class C>
__device__ __forceinline__ void node_collide_fe(C (&f)[2][L::Q], C rho, C phi, const C (&gp)[3], C lp, C omega,
                                                C omega_g, C g, C kappa, C gamma) {
    using A = Ar<C>;
    constexpr C cs2 = (C)(1.0 / 3.0);
    C j[3];
    node_momentum<L, C>(f[0], j);
    const C inv_rho = A::rcp(rho);
    C u[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) u[d] = A::mul(j[d], inv_rho);
    const C uu = L::D == 3 ? A::fma(u[0], u[0], A::fma(u[1], u[1], A::mul(u[2], u[2])))
                           : A::fma(u[0], u[0], A::mul(u[1], u[1]));
    const C gg = L::D == 3 ? A::fma(gp[0], gp[0], A::fma(gp[1], gp[1], A::mul(gp[2], gp[2])))
                           : A::fma(gp[0], gp[0], A::mul(gp[1], gp[1]));
    const C mu = A::sub(A::sub(A::mul(A::mul((C)0.5, cs2), fe_log(A::mul(A::add(rho, phi), A::rcp(A::sub(rho, phi))))),
                               A::mul(A::mul((C)0.5, A::mul(g, cs2)), phi)),
                        A::mul(kappa, lp));
    const C pb = A::fma(A::mul((C)0.25, A::mul(g, cs2)), A::mul(A::sub(rho, phi), A::add(rho, phi)), A::mul(cs2, rho));
    const C s = A::sub(A::sub(A::sub(pb, A::mul(A::mul(kappa, phi), lp)), A::mul(A::mul((C)0.5, kappa), gg)),
                       A::mul(cs2, rho));
    const C sg = A::sub(A::mul(gamma, mu), A::mul(cs2, phi));
    const C ku = A::mul(cs2, uu), kg = A::mul(cs2, gg);
    // f and g together from here on (first and second of each pair)
    using A2 = Ar2<C>;
    const Two<C> rp{rho, phi}, rp3 = A2::mul(both((C)3), rp), om{omega, omega_g}, ss{s, sg}, ku2 = both(ku);
    Two<C> u2[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) u2[d] = both(u[d]);
    SignedSumV<Two<C>> neq;  // sum_{i>0} (f^eq_i - f_i), sum_{i>0} (g^eq_i - g_i)
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        const Two<C> cu = node_cu2<L>(i, u2);
        const C cg = node_cu<L, C>(i, gp);
        int c2 = 0;
#pragma unroll
        for (int d = 0; d < L::D; ++d) c2 += L::c(i, d) * L::c(i, d);
        const C iso = (C)((double)c2 - (double)L::D / 3.0);  // c.c - D cs2
        const Two<C> quad_u = A2::sub(A2::mul_split(cu, cu), ku2);  // (c.u)^2 - cs2 u.u
        const C quad_g = A::sub(A::mul(cg, cg), kg);
        Two<C> h = A2::mul(rp, quad_u);
        h.a = A::fma(kappa, quad_g, h.a);
        h = A2::fma(ss, both(iso), h);
        const Two<C> feq = A2::mul_split(both((C)L::w(i)), A2::fma(both((C)4.5), h, A2::fma(rp3, cu, rp)));
        const Two<C> fi{f[0][i], f[1][i]};
        const Two<C> d = A2::sub(feq, fi);
        neq.add(d);
        const Two<C> n = A2::fma(om, d, fi);
        f[0][i] = n.a;
        f[1][i] = n.b;
    }
    const Two<C> n = A2::fma(om, neg2(neq.get()), Two<C>{f[0][0], f[1][0]});
    f[0][0] = n.a;
    f[1][0] = n.b;
}

// The collision of the lattice's forcing scheme, chosen at run time (kernels
// whose launch shapes accept either scheme).
template <class L, class C>
__device__ __forceinline__ void node_collide_any(int forcing, C (&f)[2][L::Q], C rA, C rB, const C (&gA)[3],
                                                 const C (&gB)[3], C omega_A, C omega_B, C tau_A, C tau_B) {
    if (forcing == kForcingGuo)
        node_collide_guo<L, C>(f, rA, rB, gA, gB, omega_A, omega_B);
    else
        node_collide<L, C>(f, rA, rB, gA, gB, omega_A, omega_B, tau_A, tau_B);
}

// The whole node update after the pulls: the SC force (and body force) with
// the lattice's forcing scheme, or the FE derivatives and collision, chosen at
// run time.  r0, r1: the two population sums of the node (rho_A, rho_B for SC;
// rho, phi for FE); nbr(i) returns the neighbour's pair of sums at x + c_i.
template <class L, class C, class Args, class Nbr>
__device__ __forceinline__ void node_update(const Args& a, int y, const Nbr& nbr, C (&f)[2][L::Q], C r0, C r1) {
    if (a.model == kModelFE) {
        C gp[3], lp;
        node_fe_derivs<L, C>(nbr, r1, gp, lp);
        node_collide_fe<L, C>(f, r0, r1, gp, lp, a.omega_A, a.omega_B, a.G, a.kappa, a.gamma);
        return;
    }
    C gA[3], gB[3];
    node_force<L, C>(nbr, a.G, gA, gB);
    node_body_force<C>(a.body_A, y, a.ny, gA, gB);
    node_collide_any<L, C>(a.forcing, f, r0, r1, gA, gB, a.omega_A, a.omega_B, a.tau_A, a.tau_B);
}

}  // namespace lbmsc

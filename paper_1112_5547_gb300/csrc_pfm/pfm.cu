// Pseudo-spectral phase-field model of Sec. 3 on one GPU (C ABI in pfm.h).
//
// One time step (Sec. 3.1, Eqs. eq10-eq13), all fields periodic:
//   1. prep (spectral, one thread per complex coefficient): phi^, i k phi^ (D
//      components), -|k|^2 phi^ and u^ (D components), scaled by 1/N, into the
//      inverse-transform batch;
//   2. one batched complex-to-real cuFFT call (2 + 2D transforms);
//   3. phys (one thread per node): u.grad phi, the explicit Cahn-Hilliard
//      bracket ln((rho+phi)/(rho-phi))/g_tau - 3 phi, the capillary force
//      mu grad phi / rho and the products u_a u_b, into the forward batch;
//   4. one batched real-to-complex cuFFT call (2 + D + D(D+1)/2 transforms);
//   5. update (spectral): S^ and the projected momentum right-hand side N^,
//      then phi^ and u^ by AB2 (explicit) / Crank-Nicolson (implicit).
// The FP64 solver does the same with its own transforms fused into three or four
// kernels a step where the sizes allow (pfm_fft.cuh); cuFFT takes FP32 and the rest.
// The spectral state (phi^, u^ and the previous explicit terms) stays in the
// caller's workspace between steps; the real fields exist only inside a step.
#include <cuda_runtime.h>
#include <cufft.h>

#include <cstdint>
#include <cstring>
#include <atomic>
#include <new>

#include "../../include/pfm.h"
#include "pfm_fft.cuh"

namespace {

constexpr double kCs2 = 1.0 / 3.0;

template <class T> struct Cx;
template <> struct Cx<float> {
    using type = cufftComplex;
};
template <> struct Cx<double> {
    using type = cufftDoubleComplex;
};

struct Geometry {
    int dim, nx, ny, nz, nxh;  // nxh = nx/2 + 1 (the half axis of the real transforms)
    long long nreal, ncplx;
    double dk[3];  // 2 pi / n of each axis
};

// Products and sums rounded as written, where several kernels form the same value.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// Wavenumbers of complex coefficient c (x the half axis, fastest): the full
// ones (Laplacian) and the first-derivative ones (Nyquist of an even axis
// zeroed), in the solver's precision T (FP32 arithmetic for the FP32 solver:
// FP64 throughput is a small fraction of FP32 on this GPU).
template <class T> struct Wave {
    T k[3], kd[3], k2;
};

// One axis: the frequency of index i of n points (the Nyquist index of an even
// axis is -n/2, as numpy's fftfreq), full and for first derivatives.
template <class T> __device__ __forceinline__ void wave_axis(const Geometry& g, int a, int i, T& k, T& kd) {
    const int n = a == 0 ? g.nx : (a == 1 ? g.ny : g.nz);
    const bool nyquist = n % 2 == 0 && i == n / 2;
    const int f = nyquist ? -n / 2 : (i <= n / 2 ? i : i - n);
    k = (T)g.dk[a] * (T)f;  // no division: FP64 ones are a dozen operations each
    kd = nyquist ? (T)0 : k;
}
template <class T> __device__ __forceinline__ Wave<T> wave_at(const Geometry& g, int ix, int iy, int iz) {
    Wave<T> w;
    wave_axis<T>(g, 0, ix, w.k[0], w.kd[0]);
    wave_axis<T>(g, 1, iy, w.k[1], w.kd[1]);
    w.k[2] = w.kd[2] = (T)0;
    if (g.dim == 3) wave_axis<T>(g, 2, iz, w.k[2], w.kd[2]);
    w.k2 = fma_rn(w.k[2], w.k[2], fma_rn(w.k[1], w.k[1], mul_rn(w.k[0], w.k[0])));
    return w;
}
template <class T> __device__ __forceinline__ Wave<T> wave_of(const Geometry& g, long long c) {
    const int ix = (int)(c % g.nxh);
    const int iy = (int)((c / g.nxh) % g.ny);
    const int iz = (int)(c / ((long long)g.nxh * g.ny));
    return wave_at<T>(g, ix, iy, iz);
}

struct Coeffs {
    double rho, g, g_tau, Dc, xi2, nu, dt, inv_n, inv_rho, inv_g_tau;
    double body_half_n;  // A N / 2: the Fourier coefficient (times -+i) of A sin(2 pi y/ny) at ky = +-1
};

template <class C, class T> __device__ __forceinline__ C cmul_i(C a, T k) {  // (i k) a
    C r;
    r.x = -k * a.y;
    r.y = k * a.x;
    return r;
}
template <class C, class T> __device__ __forceinline__ C cscale(C a, T s) {
    C r;
    r.x = s * a.x;
    r.y = s * a.y;
    return r;
}
// s a, rounded: a transform's first additions may not take the product up.
__device__ __forceinline__ double2 cscale_rn(double2 a, double s) { return double2{mul_rn(s, a.x), mul_rn(s, a.y)}; }

// 1. the inverse-transform inputs: phi^, i kd_a phi^, -k^2 phi^, u^_a (each / N)
template <class T>
__global__ void pfm_prep_kernel(Geometry g, Coeffs c, const typename Cx<T>::type* __restrict__ phi_h,
                                const typename Cx<T>::type* __restrict__ u_h, typename Cx<T>::type* __restrict__ cin) {
    using C = typename Cx<T>::type;
    const int D = g.dim;
    const T inv_n = (T)c.inv_n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < g.ncplx;
         i += (long long)gridDim.x * blockDim.x) {
        const Wave<T> w = wave_of<T>(g, i);
        const C p = phi_h[i];
        cin[i] = cscale(p, inv_n);
        for (int a = 0; a < D; ++a) cin[(1 + a) * g.ncplx + i] = cscale(cmul_i(p, w.kd[a]), inv_n);
        cin[(1 + D) * g.ncplx + i] = cscale(p, -w.k2 * inv_n);
        for (int a = 0; a < D; ++a) cin[(2 + D + a) * g.ncplx + i] = cscale(u_h[a * g.ncplx + i], inv_n);
    }
}

// The nonlinear terms of one node.  in: phi, d_a phi (D), lap phi, u_a (D);
// out: u.grad phi, bracket, F_a = mu d_a phi / rho (D), u_a u_b (a <= b).
template <class T, int D> __device__ __forceinline__ void phys_node(const Coeffs& c, const T* in, T* out) {
    const T phi = in[0], lap = in[1 + D];
    const T* const gp = in + 1;
    const T* const u = in + 2 + D;
    const T rho = (T)c.rho;
    const T lnr = log((rho + phi) / (rho - phi));
    T adv = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) adv += u[a] * gp[a];
    out[0] = adv;
    out[1] = lnr * (T)c.inv_g_tau - (T)3 * phi;
    const T mu = (T)(0.5 * kCs2) * lnr - (T)(0.5 * c.g * kCs2) * phi - (T)(0.25 * c.g * kCs2 * kCs2) * lap;
    const T mr = mu * (T)c.inv_rho;
#pragma unroll
    for (int a = 0; a < D; ++a) out[2 + a] = mr * gp[a];
    int q = 2 + D;
#pragma unroll
    for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = a; b < D; ++b) out[q++] = u[a] * u[b];
}

// 3. nonlinear terms in physical space, fields as planes of N reals.
template <class T, int D>
__global__ void pfm_phys_kernel(Geometry g, Coeffs c, const T* __restrict__ rin, T* __restrict__ rout) {
    const long long N = g.nreal;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x) {
        T in[2 + 2 * D], out[2 + D + D * (D + 1) / 2];
#pragma unroll
        for (int f = 0; f < 2 + 2 * D; ++f) in[f] = rin[f * N + n];
        phys_node<T, D>(c, in, out);
#pragma unroll
        for (int f = 0; f < 2 + D + D * (D + 1) / 2; ++f) rout[f * N + n] = out[f];
    }
}

// index of the product u_a u_b (a, b in any order) in the forward batch
__device__ __forceinline__ int uu_slot(int D, int a, int b) {
    if (a > b) {
        const int t = a;
        a = b;
        b = t;
    }
    int q = 2 + D;
    for (int i = 0; i < a; ++i) q += D - i;
    return q + (b - a);
}

// 5. The AB2 / CN update of one coefficient: phi^ and u^ from S^ without its
// implicit-split term (sx, sy = -adv^ - D k^2 bracket^) and the momentum
// right-hand side (nx, ny) before forcing and projection.  prev: S^ and N^ of the
// step before (first: none); on return s and n hold this step's.
template <class T, class C, int D>
__device__ __forceinline__ void update_coeff(const Geometry& g, const Coeffs& c, int first, const Wave<T>& w, int ix, int iy,
                                             int iz, C& p, C (&u)[D], C& s, C (&n)[D], const C& s_prev, const C (&n_prev)[D]) {
    const T Dc = (T)c.Dc, dt = (T)c.dt, nu = (T)c.nu;
    const T bi = (T)(c.Dc * (c.xi2 - c.dt * c.Dc / 2.0));
    const T half = (T)0.5, one = (T)1, three = (T)3;
    const T k2 = w.k2, k4 = mul_rn(k2, k2), bk = mul_rn(bi, k4);
    s.x = fma_rn(-bk, p.x, s.x);
    s.y = fma_rn(-bk, p.y, s.y);
    const C sp = first ? s : s_prev;
    // (a x + dt (3 s - s') / 2) / b of one component, inv = 1 / b
    auto advance = [&](T a, T x, T cur, T old, T inv) {
        return mul_rn(fma_rn(a, x, mul_rn(mul_rn(dt, fma_rn(three, cur, -old)), half)), inv);
    };
    const T lam = mul_rn(Dc, fma_rn(mul_rn(mul_rn(dt, Dc), half), k4, mul_rn((T)2, k2)));
    const T hl = mul_rn(mul_rn(dt, lam), half), am = one - hl, inv_ap = one / (one + hl);
    p = C{advance(am, p.x, s.x, sp.x, inv_ap), advance(am, p.y, s.y, sp.y, inv_ap)};
    // Kolmogorov forcing A sin(2 pi y/ny) e_x: -i A N/2 at ky = +1, +i A N/2 at ky = -1 (kx = kz = 0)
    if (c.body_half_n != 0.0 && g.ny > 2 && ix == 0 && iz == 0) {
        if (iy == 1) n[0].y -= (T)c.body_half_n;
        if (iy == g.ny - 1) n[0].y += (T)c.body_half_n;
    }
    T kd2 = 0, kre = 0, kim = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        kd2 = fma_rn(w.kd[a], w.kd[a], kd2);
        kre = fma_rn(w.kd[a], n[a].x, kre);
        kim = fma_rn(w.kd[a], n[a].y, kim);
    }
    const T inv = kd2 > (T)0 ? one / kd2 : (T)0;
    const bool mean = k2 == (T)0;
    const T hv = mul_rn(mul_rn(dt, mul_rn(nu, k2)), half), bm = one - hv, inv_bp = one / (one + hv);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        n[a] = mean ? C{(T)0, (T)0}
                    : C{fma_rn(-mul_rn(w.kd[a], kre), inv, n[a].x), fma_rn(-mul_rn(w.kd[a], kim), inv, n[a].y)};
        const C prev = first ? n[a] : n_prev[a];
        u[a] = C{advance(bm, u[a].x, n[a].x, prev.x, inv_bp), advance(bm, u[a].y, n[a].y, prev.y, inv_bp)};
    }
}

template <class T, int D>
__global__ void pfm_update_kernel(Geometry g, Coeffs c, int first, const typename Cx<T>::type* __restrict__ cout,
                                  typename Cx<T>::type* __restrict__ phi_h, typename Cx<T>::type* __restrict__ u_h,
                                  typename Cx<T>::type* __restrict__ s_prev, typename Cx<T>::type* __restrict__ n_prev) {
    using C = typename Cx<T>::type;
    const long long M = g.ncplx;
    const T Dc = (T)c.Dc;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < M; i += (long long)gridDim.x * blockDim.x) {
        const int ix = (int)(i % g.nxh), iy = (int)((i / g.nxh) % g.ny), iz = (int)(i / ((long long)g.nxh * g.ny));
        const Wave<T> w = wave_at<T>(g, ix, iy, iz);
        const C adv = cout[i], br = cout[M + i];
        C p = phi_h[i], u[D], n[D], np[D], sp{(T)0, (T)0};
        C s{-adv.x - Dc * w.k2 * br.x, -adv.y - Dc * w.k2 * br.y};
        if (!first) sp = s_prev[i];
        // momentum right-hand side: -i sum_b kd_b (u_a u_b)^ + F_a^
#pragma unroll
        for (int a = 0; a < D; ++a) {
            T re = cout[(2 + a) * M + i].x, im = cout[(2 + a) * M + i].y;
#pragma unroll
            for (int b = 0; b < D; ++b) {
                const C q = cout[uu_slot(D, a, b) * M + i];
                // -(i kd_b) q = kd_b (q.y - i q.x)
                re += w.kd[b] * q.y;
                im -= w.kd[b] * q.x;
            }
            n[a] = C{re, im};
            np[a] = first ? C{(T)0, (T)0} : n_prev[a * M + i];
            u[a] = u_h[a * M + i];
        }
        update_coeff<T, C, D>(g, c, first, w, ix, iy, iz, p, u, s, n, sp, np);
        phi_h[i] = p;
        s_prev[i] = s;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            u_h[a * M + i] = u[a];
            n_prev[a * M + i] = n[a];
        }
    }
}

// ---- the FP64 step with the transforms inside (pfm_fft.cuh) -------------------

using pfm_fft::R0;

struct State {
    using C = double2;
    C* phi;
    C* u;
    C* s_prev;
    C* n_prev;
};

constexpr int kColThreads = 512;

// The spectral axis (z in 3D, y in 2D), M columns of x at one y (3D).  FWD: the
// fields of `in` (adv, bracket, G_a, H_a; H_a the stress (u_a u_last)^ whose
// derivative along this axis is still to be taken) are transformed and the state is
// advanced.  INV: phi, its derivative along this axis, its second one and u go out.
// in may be out: a block reads its own columns of every field before it writes.
// Its arithmetic outside the transforms is rounded as written (mul_rn, fma_rn), so a
// step gives the same bits whether it is the first of a call, in the middle or the
// last: left to the compiler, the three kernels contracted different pairs.
template <int D, bool FWD, bool INV>
__global__ void __launch_bounds__(kColThreads)
    pfm_spectral_kernel(Geometry g, Coeffs c, pfm_fft::Plan plan, const double2* __restrict__ tw, int M,
                        int first, const double2* in, double2* out,
                        State st) {
    using C = double2;
    using T = double;
    extern __shared__ __align__(16) unsigned char pfm_smem[];
    pfm_fft::Columns col(plan, tw, pfm_smem, M);
    const int ix = blockIdx.x * M + col.x, iy3 = D == 3 ? (int)blockIdx.y : 0;
    const bool on = ix < g.nxh;
    const long long F = g.ncplx, stride = D == 3 ? (long long)g.nxh * g.ny : g.nxh;
    const long long base = ix + (long long)g.nxh * iy3;
    auto at = [&](int q) { return base + stride * col.row(q); };
    auto load = [&](const C* f, C (&v)[R0]) {
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = on ? f[at(q)] : C{(T)0, (T)0};
    };
    C p[R0], n[D][R0];  // phi; the momentum right-hand side, then u
    if (FWD) {
        C s[R0], v[R0];
        load(in, v);
        col.run(v);
#pragma unroll
        for (int q = 0; q < R0; ++q) s[q] = C{-v[q].x, -v[q].y};
        load(in + F, v);
        col.run(v);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const Wave<T> w = D == 3 ? wave_at<T>(g, ix, iy3, col.row(q)) : wave_at<T>(g, ix, col.row(q), 0);
            const T dk = mul_rn((T)c.Dc, w.k2);
            s[q].x = fma_rn(-dk, v[q].x, s[q].x);
            s[q].y = fma_rn(-dk, v[q].y, s[q].y);
        }
#pragma unroll
        for (int a = 0; a < D; ++a) {
            load(in + (2 + a) * F, n[a]);
            col.run(n[a]);
            load(in + (2 + D + a) * F, v);
            col.run(v);
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                T k, kd;
                wave_axis<T>(g, D - 1, col.row(q), k, kd);
                n[a][q].x = fma_rn(kd, v[q].y, n[a][q].x);
                n[a][q].y = fma_rn(-kd, v[q].x, n[a][q].y);
            }
        }
        load(st.phi, p);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            const int iy = D == 3 ? iy3 : col.row(q), iz = D == 3 ? col.row(q) : 0;
            const Wave<T> w = wave_at<T>(g, ix, iy, iz);
            const long long i = at(q);
            C uu[D], nn[D], np[D], sp{(T)0, (T)0};
            if (on && !first) sp = st.s_prev[i];
#pragma unroll
            for (int a = 0; a < D; ++a) {
                uu[a] = on ? st.u[a * F + i] : C{(T)0, (T)0};
                nn[a] = n[a][q];
                np[a] = on && !first ? st.n_prev[a * F + i] : C{(T)0, (T)0};
            }
            update_coeff<T, C, D>(g, c, first, w, ix, iy, iz, p[q], uu, s[q], nn, sp, np);
#pragma unroll
            for (int a = 0; a < D; ++a) n[a][q] = uu[a];
            if (on) {
                st.phi[i] = p[q];
                st.s_prev[i] = s[q];
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    st.u[a * F + i] = uu[a];
                    st.n_prev[a * F + i] = nn[a];
                }
            }
        }
    } else {
        load(st.phi, p);
#pragma unroll
        for (int a = 0; a < D; ++a) load(st.u + a * F, n[a]);
    }
    if (INV) {
        const T inv_n = (T)c.inv_n;
        C v[R0];
        auto send = [&](int f) {
            col.run_inverse(v);
#pragma unroll
            for (int q = 0; q < R0; ++q)
                if (on) out[f * F + at(q)] = v[q];
        };
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = p[q] = cscale_rn(p[q], inv_n);
        send(0);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            T k, kd;
            wave_axis<T>(g, D - 1, col.row(q), k, kd);
            v[q] = C{mul_rn(-kd, p[q].y), mul_rn(kd, p[q].x)};
        }
        send(1);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            T k, kd;
            wave_axis<T>(g, D - 1, col.row(q), k, kd);
            v[q] = cscale_rn(p[q], -k * k);
        }
        send(2);
#pragma unroll
        for (int a = 0; a < D; ++a) {
#pragma unroll
            for (int q = 0; q < R0; ++q) v[q] = cscale_rn(n[a][q], inv_n);
            send(3 + a);
        }
    }
}

// y in 3D, inverse: phi, d_z phi, lap phi so far, u come in; phi, d_y phi, d_z phi,
// lap phi (with y's part) and u go out.  blockIdx.y is z.
__global__ void __launch_bounds__(kColThreads)
    pfm_y_inverse_kernel(Geometry g, pfm_fft::Plan plan, const double2* __restrict__ tw, int M,
                         const double2* __restrict__ in, double2* __restrict__ out) {
    using C = double2;
    using T = double;
    extern __shared__ __align__(16) unsigned char pfm_smem[];
    pfm_fft::Columns col(plan, tw, pfm_smem, M);
    const int ix = blockIdx.x * M + col.x;
    const bool on = ix < g.nxh;
    const long long F = g.ncplx, base = ix + (long long)g.nxh * g.ny * blockIdx.y;
    auto at = [&](int q) { return base + (long long)g.nxh * col.row(q); };
    auto load = [&](int f, C (&v)[R0]) {
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = on ? in[f * F + at(q)] : C{(T)0, (T)0};
    };
    // the next field's loads are in flight while one is transformed
    C p[R0], v[R0], w[R0];
    auto send = [&](int f) {
        col.run_inverse(v);
#pragma unroll
        for (int q = 0; q < R0; ++q)
            if (on) out[f * F + at(q)] = v[q];
    };
    auto next = [&]() {
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = w[q];
    };
    load(0, p);
    load(2, w);
#pragma unroll
    for (int q = 0; q < R0; ++q) v[q] = p[q];
    send(0);
#pragma unroll
    for (int q = 0; q < R0; ++q) {
        T k, kd;
        wave_axis<T>(g, 1, col.row(q), k, kd);
        v[q] = cmul_i(p[q], kd);
    }
    send(1);
#pragma unroll
    for (int q = 0; q < R0; ++q) {
        T k, kd;
        wave_axis<T>(g, 1, col.row(q), k, kd);
        v[q] = C{w[q].x - k * k * p[q].x, w[q].y - k * k * p[q].y};
    }
    load(1, w);
    send(3);
    next();
    load(3, w);
    send(2);
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        next();
        if (a < 2) load(4 + a, w);
        send(4 + a);
    }
}

// y in 3D, forward: adv, bracket, G_a, u_x u_y, u_x u_z, u_y u_y, u_y u_z, u_z u_z
// come in; adv, bracket, G_a - i k_y (u_a u_y)^ and H_a = (u_a u_z)^ go out.
__global__ void __launch_bounds__(kColThreads)
    pfm_y_forward_kernel(Geometry g, pfm_fft::Plan plan, const double2* __restrict__ tw, int M,
                         const double2* __restrict__ in, double2* __restrict__ out) {
    using C = double2;
    using T = double;
    extern __shared__ __align__(16) unsigned char pfm_smem[];
    pfm_fft::Columns col(plan, tw, pfm_smem, M);
    const int ix = blockIdx.x * M + col.x;
    const bool on = ix < g.nxh;
    const long long F = g.ncplx, base = ix + (long long)g.nxh * g.ny * blockIdx.y;
    auto at = [&](int q) { return base + (long long)g.nxh * col.row(q); };
    // the next field's loads are in flight while one is transformed
    C v[R0], h[R0], w[R0];
    auto load = [&](int f) {
#pragma unroll
        for (int q = 0; q < R0; ++q) w[q] = on ? in[f * F + at(q)] : C{(T)0, (T)0};
    };
    auto take = [&](C (&x)[R0], int following) {
#pragma unroll
        for (int q = 0; q < R0; ++q) x[q] = w[q];
        if (following >= 0) load(following);
        col.run(x);
    };
    auto send = [&](int f, const C (&x)[R0]) {
#pragma unroll
        for (int q = 0; q < R0; ++q)
            if (on) out[f * F + at(q)] = x[q];
    };
    load(0);
    take(v, 1);
    send(0, v);
    take(v, 6);
    send(1, v);
    take(v, 9);
    send(5, v);
    take(v, 5);
    send(7, v);
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        take(h, 2 + a);            // u_a u_y
        if (a == 2) send(6, h);    // u_y u_z is H_y too
        take(v, a < 2 ? 7 + a : -1);
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            T k, kd;
            wave_axis<T>(g, 1, col.row(q), k, kd);
            v[q].x += kd * h[q].y;
            v[q].y -= kd * h[q].x;
        }
        send(2 + a, v);
    }
}

// x: R rows per block, all fields of the rows in shared memory at once, each line
// a half-length complex one (m = nx / 2).  In: phi, d_y phi (d_z phi), lap phi so
// far, u; d_x phi and x's part of lap phi are formed from phi.  Out: adv, bracket,
// F_a - i k_x (u_a u_x)^ and the other stresses.
constexpr int kRowThreads = 256;
__host__ __device__ constexpr int x_in_fields(int D) { return 2 + 2 * D; }
__host__ __device__ constexpr int x_out_fields(int D) { return 2 + D + D * (D + 1) / 2; }
__host__ __device__ inline int x_pitch(int m) { return m + m / 16 + 1; }  // a shift of one value every 16
inline size_t x_smem(int nx, int D, int R) {
    return ((size_t)2 * x_out_fields(D) * R * x_pitch(nx / 2) + nx + nx / 4 + 1) * sizeof(double2);
}

template <int D>
__global__ void __launch_bounds__(kRowThreads, 2)
    pfm_x_kernel(Geometry g, Coeffs c, pfm_fft::Plan plan, const double2* __restrict__ gtw, int R,
                 const double2* __restrict__ in, double2* __restrict__ out) {
    using C = double2;
    using T = double;
    constexpr int NI = x_in_fields(D), NO = x_out_fields(D);
    static_assert(NO >= NI, "the buffers hold either set of fields");
    extern __shared__ __align__(16) unsigned char pfm_smem[];
    const int tid = threadIdx.x, nt = kRowThreads;
    const int m = plan.n, pitch = x_pitch(m), nb = m / R0;
    const long long F = g.ncplx, rows = (long long)g.ny * g.nz, row0 = (long long)blockIdx.x * R;
    C* a = reinterpret_cast<C*>(pfm_smem);
    C* b = a + (size_t)NO * R * pitch;
    C* const tw = b + (size_t)NO * R * pitch;     // e^{-2 pi i t / nx}
    T* const kxs = reinterpret_cast<T*>(tw + g.nx);  // wavenumbers 0 .. m
    for (int k = tid; k < g.nx; k += nt) tw[k] = gtw[k];
    for (int k = tid; k <= m; k += nt) {
        T kd;
        wave_axis<T>(g, 0, k, kxs[k], kd);
    }
    __syncthreads();
    auto at = [pitch](int l, int i) { return l * pitch + pfm_fft::pad16(i); };

    // inverse: Z_k = (X_k + conj X_{m-k}) + i e^{2 pi i k / nx} (X_k - conj X_{m-k}); its
    // inverse transform holds the samples 2 j and 2 j + 1
    pfm_fft::for_rows(nb, NI * R, tid, nt, [&](int j, int l0, int par) {
        for (int l = l0; l < NI * R; l += par) {
            const int f = l / R;
            const long long row = row0 + (l - f * R);
            const bool on = row < rows;
            const C* const phi = in + row * g.nxh;
            const C* const own = f < 2 ? phi : phi + (f - 1) * F;
            C x[R0], y[R0];
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const int k = j + q * nb;
                x[q] = on ? own[k] : C{(T)0, (T)0};
                y[q] = on ? own[m - k] : C{(T)0, (T)0};
            }
            if (f == 1) {  // d_x phi (no first derivative at the Nyquist mode)
#pragma unroll
                for (int q = 0; q < R0; ++q) {
                    const int k = j + q * nb;
                    x[q] = cmul_i(x[q], kxs[k]);
                    y[q] = cmul_i(y[q], k == 0 ? (T)0 : kxs[m - k]);
                }
            } else if (f == 1 + D) {  // x's part of lap phi
#pragma unroll
                for (int q = 0; q < R0; ++q) {
                    const int k = j + q * nb;
                    const C u = on ? phi[k] : C{(T)0, (T)0}, v = on ? phi[m - k] : C{(T)0, (T)0};
                    const T ku = kxs[k] * kxs[k], kv = kxs[m - k] * kxs[m - k];
                    x[q] = C{x[q].x - ku * u.x, x[q].y - ku * u.y};
                    y[q] = C{y[q].x - kv * v.x, y[q].y - kv * v.y};
                }
            }
            if (j == 0) x[0].y = y[0].y = (T)0;  // the two real coefficients
            C v[R0];
#pragma unroll
            for (int q = 0; q < R0; ++q) {
                const C yc = pfm_fft::cnj(y[q]);
                const C d = pfm_fft::mul(pfm_fft::sub(x[q], yc), pfm_fft::cnj(tw[j + q * nb]));
                v[q] = C{x[q].y + yc.y + d.x, x[q].x + yc.x - d.y};  // exchanged: an inverse transform
            }
            pfm_fft::dft<R0>(v);
#pragma unroll
            for (int q = 0; q < R0; ++q) a[at(l, j * R0 + q)] = v[q];
        }
    });
    __syncthreads();
    C* src = pfm_fft::middle_rows(a, b, plan, NI * R, pitch, tid, nt, tw);
    C* dst = src == a ? b : a;
    pfm_fft::pass_rows<R0>(src, dst, m, NI * R, pitch, nb, tid, nt, tw, true);
    __syncthreads();
    // nonlinear terms of two neighbouring nodes at a time
#pragma unroll 1
    for (int w = tid; w < R * m; w += nt) {
        const int r = w / m, i = w - r * m;
        T x0[NI], x1[NI], y0[NO], y1[NO];
#pragma unroll
        for (int f = 0; f < NI; ++f) {
            const C v = dst[at(f * R + r, i)];
            x0[f] = v.x;
            x1[f] = v.y;
        }
        phys_node<T, D>(c, x0, y0);
        phys_node<T, D>(c, x1, y1);
#pragma unroll
        for (int f = 0; f < NO; ++f) src[at(f * R + r, i)] = C{y0[f], y1[f]};
    }
    __syncthreads();
    // forward
    pfm_fft::for_rows(nb, NO * R, tid, nt, [&](int j, int l0, int par) {
        for (int l = l0; l < NO * R; l += par) {
            C v[R0];
#pragma unroll
            for (int q = 0; q < R0; ++q) v[q] = src[at(l, j + q * nb)];
            pfm_fft::dft<R0>(v);
#pragma unroll
            for (int q = 0; q < R0; ++q) dst[at(l, j * R0 + q)] = v[q];
        }
    });
    __syncthreads();
    src = pfm_fft::middle_rows(dst, src, plan, NO * R, pitch, tid, nt, tw);
    dst = src == a ? b : a;
    pfm_fft::pass_rows<R0>(src, dst, m, NO * R, pitch, nb, tid, nt, tw);
    __syncthreads();
    // X_k = (Z_k + conj Z_{m-k}) / 2 - i/2 e^{-2 pi i k / nx} (Z_k - conj Z_{m-k}), Z_m = Z_0
#pragma unroll 1
    for (int w = tid; w < R * (m + 1); w += nt) {
        const int r = w / (m + 1), k = w - r * (m + 1);
        const long long row = row0 + r;
        if (row >= rows) continue;
        const int k0 = k == m ? 0 : k, k1 = k == 0 ? 0 : m - k;
        const C t = tw[k];
        const T kd = k == m ? (T)0 : kxs[k];
        auto spec = [&](int f) -> C {
            const C z = dst[at(f * R + r, k0)], y = pfm_fft::cnj(dst[at(f * R + r, k1)]);
            const C d = pfm_fft::mul(pfm_fft::sub(z, y), t);
            return C{(T)0.5 * (z.x + y.x + d.y), (T)0.5 * (z.y + y.y - d.x)};
        };
        C* const o = out + row * g.nxh + k;
        o[0] = spec(0);
        o[F] = spec(1);
        int e = 2 + D;
#pragma unroll
        for (int b2 = 0; b2 < D; ++b2) {  // F_b - i k_x (u_x u_b)^
            C v = spec(2 + b2);
            const C h = spec(2 + D + b2);
            v.x += kd * h.y;
            v.y -= kd * h.x;
            o[(2 + b2) * F] = v;
            if (b2 > 0) o[(e++) * F] = h;
        }
#pragma unroll
        for (int f = 2 + 2 * D; f < NO; ++f) o[(e++) * F] = spec(f);
    }
}

constexpr size_t kFusedSmem = 200 * 1024;  // dynamic shared memory a fused kernel may use (bytes)

// Shapes of the fused kernels.  They take FP64, even nx whose half, and ny and nz, are
// 16 times factors 2, 3, 4, 5, up to the lengths whose lines fit shared memory, and the
// boxes that give the blocks of every axis enough SMs to run on (fused_pays); other
// sizes go through cuFFT (ok = false).
struct Fused {
    bool ok;
    pfm_fft::Plan x, y, z;
    int My, Mz, R;  // columns per block of the y and z kernels, rows per block of x
};

// Columns per block of an axis of n points: whole 64-byte segments of a row where
// the block's threads allow it, narrower where that leaves SMs without a block
// (512 x 512 FP64: 129 blocks of two columns instead of 65 of four).
inline int fused_columns(const pfm_fft::Plan& p, int nxh, long long lines) {
    int M = 4;
    while (M > 1 && (p.n / R0) * M > kColThreads) M /= 2;
    while (M > 2 && (nxh + M - 1) / M * lines < 152) M /= 2;
    return M;
}

// Whether the fused kernels are faster than the batched transforms: a block's chain
// of transforms is longer than the batched ones' launches, and its axis' blocks are
// few where the box is small or narrow.  Measured (GB300, us a step, batched / fused):
//   2D, 98304 nodes: 96 x 960 (just below) 218 / 183, 128 x 768 209 / 161; fewer: 128 x 512 127 / 130, 256 x 256 123 / 136,
//       64 x 1024 133 / 160, 16 x 960 78 / 148
//   2D, nx > 256 (more than 64 blocks of two columns): 400 x 288 248 / 223, 1024 x 288 545 / 489; narrower:
//       1024 x 256 444 / 447, 384 x 256 191 / 189, 1024 x 128 321 / 376, 640 x 128 178 / 256
//   2D, nx <= 1024: 512 x 1024 852 / 659; longer (the row kernel's first pass has 160 butterflies for its 256 threads
//       at 1280, and one block an SM): 512 x 1280 993 / 1063, 1024 x 1280 2021 / 1795, 48 x 1440 150 / 232
//   3D, 131072 nodes: 32 x 64 x 64 265 / 243; fewer: 32^3 118 / 164
//   3D, nx >= 64: 512 x 32 x 64 1938 / 1672; narrower: 512 x 32 x 32 951 / 1181, 64 x 64 x 32 259 / 278
//   3D, nz >= 32 (16 leave a block of the z kernel half a warp) unless rows are longer:
//       16 x 96 x 96 361 / 352, 16 x 512 x 64 961 / 1011, 16 x 128 x 64 275 / 293
inline bool fused_pays(const Geometry& g) {
    if (g.dim == 2) return g.nreal >= 98304 && g.nx > 256 && g.nx <= 1024;
    return g.nreal >= 131072 && g.nx >= 64 && (g.nz >= 32 || g.nx >= 96);
}

Fused fused_shape(const Geometry& g, bool fp64) {
    Fused f;
    memset(&f, 0, sizeof(f));
    const size_t smem = kFusedSmem;
    if (!fp64 || g.nx % 2 != 0 || g.ny > 1024 || g.nz > 1024 || !fused_pays(g)) return f;
    if (!pfm_fft::make_plan(g.nx / 2, &f.x) || !pfm_fft::make_plan(g.ny, &f.y)) return f;
    if (g.dim == 3 && !pfm_fft::make_plan(g.nz, &f.z)) return f;
    f.My = fused_columns(f.y, g.nxh, g.nz);
    f.Mz = g.dim == 3 ? fused_columns(f.z, g.nxh, g.ny) : 0;
    const int D = g.dim, points = x_in_fields(D) * (g.nx / 2);
    const long long rows = (long long)g.ny * g.nz;
    f.R = (kRowThreads * R0 + points - 1) / points;  // a first radix for every thread
    if (f.R > 8) f.R = 8;
    while (f.R > 1 && rows / f.R < 304) f.R /= 2;
    if (x_smem(g.nx, D, f.R) > smem || pfm_fft::columns_smem(g.ny, f.My) > smem ||
        (g.dim == 3 && pfm_fft::columns_smem(g.nz, f.Mz) > smem))
        return f;
    f.ok = true;
    return f;
}

constexpr size_t kAlign = 256;
size_t align_up(size_t b) { return (b + kAlign - 1) / kAlign * kAlign; }

bool valid(const pfm_params* p) {
    if (!p) return false;
    if (p->dim != 2 && p->dim != 3) return false;
    if (p->precision != PFM_F64 && p->precision != PFM_F32) return false;
    if (p->nx < 2 || p->ny < 2 || p->nz < 1) return false;
    if (p->dim == 2 && p->nz != 1) return false;
    if (p->dim == 3 && p->nz < 2) return false;
    if ((long long)p->nx * p->ny * p->nz >= (1LL << 31)) return false;
    // g > 0: the explicit bracket carries 1/g_tau and the mobility D = M g_tau cs2/2
    if (!(p->rho > 0) || !(p->tau > 0.5) || !(p->dt > 0) || !(p->g > 0) || !(p->g - p->g == 0.0)) return false;
    if (!(p->body_A - p->body_A == 0.0)) return false;
    return true;
}

Geometry geometry(const pfm_params* p) {
    Geometry g;
    g.dim = p->dim;
    g.nx = p->nx;
    g.ny = p->ny;
    g.nz = p->dim == 3 ? p->nz : 1;
    g.nxh = p->nx / 2 + 1;
    g.nreal = (long long)g.nx * g.ny * g.nz;
    g.ncplx = (long long)g.nxh * g.ny * g.nz;
    g.dk[0] = 6.283185307179586 / g.nx;
    g.dk[1] = 6.283185307179586 / g.ny;
    g.dk[2] = 6.283185307179586 / g.nz;
    return g;
}

int n_inverse(int D) { return 2 + 2 * D; }
int n_forward(int D) { return 2 + D + D * (D + 1) / 2; }

struct Layout {
    size_t phi_h, u_h, s_prev, n_prev, cin, rin, rphys, cout, tw[3], total;
};

Layout layout(const Geometry& g, size_t real_bytes) {
    const size_t cb = 2 * real_bytes;
    const int D = g.dim;
    Layout L;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += align_up(bytes);
        return at;
    };
    L.phi_h = take(g.ncplx * cb);
    L.u_h = take(D * g.ncplx * cb);
    L.s_prev = take(g.ncplx * cb);
    L.n_prev = take(D * g.ncplx * cb);
    L.cin = take(n_inverse(D) * g.ncplx * cb);
    L.rin = take(n_inverse(D) * g.nreal * real_bytes);
    L.rphys = take(n_forward(D) * g.nreal * real_bytes);
    L.cout = take(n_forward(D) * g.ncplx * cb);
    // twiddle tables of the fused FP64 kernels
    L.tw[0] = take(g.nx * cb);
    L.tw[1] = take(g.ny * cb);
    L.tw[2] = take(g.nz * cb);
    L.total = o;
    return L;
}

}  // namespace

struct pfm_handle {
    pfm_params params;
    Geometry g;
    Coeffs c;
    Layout L;
    unsigned char* ws;
    cudaStream_t stream;
    cufftHandle inv, fwd;
    Fused fused;
    int started;  // an explicit term of the previous step exists
};

namespace {

Coeffs coeffs(const pfm_params* p, const Geometry& g) {
    Coeffs c;
    c.rho = p->rho;
    c.g = p->g;
    c.g_tau = p->tau * p->g / (p->tau - 0.5);
    const double M = p->rho * (p->tau - 0.5);
    c.Dc = M * c.g_tau * kCs2 / 2.0;
    c.xi2 = kCs2 / 2.0;
    c.nu = kCs2 * (p->tau - 0.5);
    c.dt = p->dt;
    c.inv_n = 1.0 / (double)g.nreal;
    c.inv_rho = 1.0 / c.rho;
    c.inv_g_tau = 1.0 / c.g_tau;
    c.body_half_n = p->body_A * (double)g.nreal / 2.0;
    return c;
}

lbm_status make_plan(const Geometry& g, bool inverse, bool dbl, int batch, cufftHandle* out) {
    int n[3];
    int rank = g.dim;
    if (g.dim == 3) {
        n[0] = g.nz;
        n[1] = g.ny;
        n[2] = g.nx;
    } else {
        n[0] = g.ny;
        n[1] = g.nx;
    }
    const cufftType t = inverse ? (dbl ? CUFFT_Z2D : CUFFT_C2R) : (dbl ? CUFFT_D2Z : CUFFT_R2C);
    if (cufftPlanMany(out, rank, n, nullptr, 1, 0, nullptr, 1, 0, t, batch) != CUFFT_SUCCESS) return LBM_ERR_CUDA;
    return LBM_OK;
}

unsigned grid_for(long long n) {
    long long b = (n + 255) / 256;
    if (b > 152LL * 32) b = 152LL * 32;
    return (unsigned)(b < 1 ? 1 : b);
}

template <class T> lbm_status exec(cufftHandle plan, bool inverse, void* in, void* out) {
    cufftResult r;
    if constexpr (sizeof(T) == 8) {
        r = inverse ? cufftExecZ2D(plan, (cufftDoubleComplex*)in, (cufftDoubleReal*)out)
                    : cufftExecD2Z(plan, (cufftDoubleReal*)in, (cufftDoubleComplex*)out);
    } else {
        r = inverse ? cufftExecC2R(plan, (cufftComplex*)in, (cufftReal*)out)
                    : cufftExecR2C(plan, (cufftReal*)in, (cufftComplex*)out);
    }
    return r == CUFFT_SUCCESS ? LBM_OK : LBM_ERR_CUDA;
}

template <class T> lbm_status step_typed(pfm_handle* h) {
    using C = typename Cx<T>::type;
    unsigned char* w = h->ws;
    const Geometry& g = h->g;
    auto P = [&](size_t off) { return (void*)(w + off); };
    pfm_prep_kernel<T><<<grid_for(g.ncplx), 256, 0, h->stream>>>(g, h->c, (const C*)P(h->L.phi_h),
                                                                 (const C*)P(h->L.u_h), (C*)P(h->L.cin));
    if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
    lbm_status s = exec<T>(h->inv, true, P(h->L.cin), P(h->L.rin));
    if (s != LBM_OK) return s;
    if (g.dim == 3)
        pfm_phys_kernel<T, 3><<<grid_for(g.nreal), 256, 0, h->stream>>>(g, h->c, (const T*)P(h->L.rin), (T*)P(h->L.rphys));
    else
        pfm_phys_kernel<T, 2><<<grid_for(g.nreal), 256, 0, h->stream>>>(g, h->c, (const T*)P(h->L.rin), (T*)P(h->L.rphys));
    if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
    s = exec<T>(h->fwd, false, P(h->L.rphys), P(h->L.cout));
    if (s != LBM_OK) return s;
    auto update = g.dim == 3 ? pfm_update_kernel<T, 3> : pfm_update_kernel<T, 2>;
    update<<<grid_for(g.ncplx), 256, 0, h->stream>>>(g, h->c, h->started ? 0 : 1, (const C*)P(h->L.cout),
                                                     (C*)P(h->L.phi_h), (C*)P(h->L.u_h), (C*)P(h->L.s_prev),
                                                     (C*)P(h->L.n_prev));
    if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
    h->started = 1;
    return LBM_OK;
}

// The fused kernels may use kFusedSmem bytes of dynamic shared memory: asked for
// once per kernel and device, never less, so that solvers of several sizes may be
// stepped from several threads (the limit belongs to the kernel, not to a launch).
template <auto Kern> cudaError_t fused_smem_once() {
    constexpr int kMaxDevices = 64;
    static std::atomic<int> done[kMaxDevices];  // zero-initialised: not yet set
    int dev = 0;
    const cudaError_t d = cudaGetDevice(&dev);
    if (d != cudaSuccess) return d;
    const bool known = dev >= 0 && dev < kMaxDevices;
    if (known && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmem);
    if (e == cudaSuccess && known) done[dev].store(1, std::memory_order_release);
    return e;
}

template <auto Kern> lbm_status launch_fused(dim3 grid, int threads, size_t smem, cudaStream_t st, void** args) {
    if (fused_smem_once<Kern>() != cudaSuccess) return LBM_ERR_CUDA;
    return cudaLaunchKernel((const void*)Kern, grid, dim3(threads), args, smem, st) == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

// Fused steps: the spectral axis sends the state inwards, then per step y, x, y
// (3D) or x (2D) and the spectral axis, which advances the state and sends it on.
template <int D> struct FusedRun {
    using C = double2;
    pfm_handle* h;
    C* at(size_t off) const { return (C*)(h->ws + off); }

    template <bool FWD, bool INV> lbm_status spectral(C* in, C* out) const {
        const Geometry& g = h->g;
        const pfm_fft::Plan& p = D == 3 ? h->fused.z : h->fused.y;
        int M = D == 3 ? h->fused.Mz : h->fused.My;
        int first = h->started ? 0 : 1;
        C* tw = at(h->L.tw[D - 1]);
        State st{at(h->L.phi_h), at(h->L.u_h), at(h->L.s_prev), at(h->L.n_prev)};
        const dim3 grid((unsigned)((g.nxh + M - 1) / M), D == 3 ? (unsigned)g.ny : 1u);
        void* args[] = {&h->g, &h->c, (void*)&p, &tw, &M, &first, &in, &out, &st};
        return launch_fused<pfm_spectral_kernel<D, FWD, INV>>(grid, p.n / R0 * M, pfm_fft::columns_smem(p.n, M), h->stream,
                                                              args);
    }
    lbm_status y(bool inverse, C* in, C* out) const {
        const Geometry& g = h->g;
        const pfm_fft::Plan& p = h->fused.y;
        int M = h->fused.My;
        C* tw = at(h->L.tw[1]);
        const dim3 grid((unsigned)((g.nxh + M - 1) / M), (unsigned)g.nz);
        void* args[] = {&h->g, (void*)&p, &tw, &M, &in, &out};
        const size_t smem = pfm_fft::columns_smem(p.n, M);
        return inverse ? launch_fused<pfm_y_inverse_kernel>(grid, p.n / R0 * M, smem, h->stream, args)
                       : launch_fused<pfm_y_forward_kernel>(grid, p.n / R0 * M, smem, h->stream, args);
    }
    lbm_status x(C* in, C* out) const {
        const Geometry& g = h->g;
        int R = h->fused.R;
        C* tw = at(h->L.tw[0]);
        const long long rows = (long long)g.ny * g.nz;
        const dim3 grid((unsigned)((rows + R - 1) / R));
        void* args[] = {&h->g, &h->c, &h->fused.x, &tw, &R, &in, &out};
        return launch_fused<pfm_x_kernel<D>>(grid, kRowThreads, x_smem(g.nx, D, R), h->stream, args);
    }
    lbm_status run(int nsteps) const {
        C* const cin = at(h->L.cin);
        C* const cout = at(h->L.cout);
        C* const mid = at(h->L.rphys);  // 10 spectral fields in the room of 11 real ones (nx >= 64)
        lbm_status s = spectral<false, true>(cin, cin);
        for (int k = 0; k < nsteps && s == LBM_OK; ++k) {
            C* back = cout;
            if constexpr (D == 3) {
                s = y(true, cin, cout);
                if (s == LBM_OK) s = x(cout, mid);
                if (s == LBM_OK) s = y(false, mid, cin);
                back = cin;
            } else {
                s = x(cin, cout);
            }
            if (s == LBM_OK) s = k + 1 < nsteps ? spectral<true, true>(back, cin) : spectral<true, false>(back, cin);
            if (s == LBM_OK) h->started = 1;
        }
        return s;
    }
};

size_t real_bytes(const pfm_params* p) { return p->precision == PFM_F64 ? 8 : 4; }

}  // namespace

extern "C" {

LBM_SC_API size_t pfm_workspace_bytes(const pfm_params* p) {
    if (!valid(p)) return 0;
    return layout(geometry(p), real_bytes(p)).total;
}

LBM_SC_API lbm_status pfm_create(const pfm_params* p, void* d_ws, size_t bytes, void* stream, pfm_handle** out) {
    if (!out) return LBM_ERR_INVALID_ARG;
    *out = nullptr;
    if (!valid(p) || !d_ws || ((uintptr_t)d_ws % kAlign) != 0) return LBM_ERR_INVALID_ARG;
    const Geometry g = geometry(p);
    const Layout L = layout(g, real_bytes(p));
    if (bytes < L.total) return LBM_ERR_OUT_OF_MEMORY;
    pfm_handle* h = new (std::nothrow) pfm_handle;
    if (!h) return LBM_ERR_OUT_OF_MEMORY;
    h->params = *p;
    h->g = g;
    h->c = coeffs(p, g);
    h->L = L;
    h->ws = static_cast<unsigned char*>(d_ws);
    h->stream = static_cast<cudaStream_t>(stream);
    h->started = 0;
    const bool dbl = p->precision == PFM_F64;
    if (make_plan(g, true, dbl, n_inverse(g.dim), &h->inv) != LBM_OK) {
        delete h;
        return LBM_ERR_CUDA;
    }
    if (make_plan(g, false, dbl, n_forward(g.dim), &h->fwd) != LBM_OK) {
        cufftDestroy(h->inv);
        delete h;
        return LBM_ERR_CUDA;
    }
    if (cufftSetStream(h->inv, h->stream) != CUFFT_SUCCESS || cufftSetStream(h->fwd, h->stream) != CUFFT_SUCCESS) {
        cufftDestroy(h->inv);
        cufftDestroy(h->fwd);
        delete h;
        return LBM_ERR_CUDA;
    }
    h->fused = fused_shape(g, dbl);
    *out = h;
    return LBM_OK;
}

LBM_SC_API lbm_status pfm_init(pfm_handle* h, const void* d_phi, const void* d_u) {
    if (!h || !d_phi) return LBM_ERR_INVALID_ARG;
    const Geometry& g = h->g;
    const int D = g.dim;
    const size_t rb = real_bytes(&h->params), cb = 2 * rb;
    unsigned char* w = h->ws;
    if (h->fused.ok) {
        const int n[3] = {g.nx, g.ny, g.nz};
        for (int a = 0; a < D; ++a)
            pfm_fft::twiddle_kernel<<<4, 256, 0, h->stream>>>((double2*)(w + h->L.tw[a]), n[a]);
        if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
    }
    // the forward batch's inputs: phi, u_a, the rest zero; transformed together
    if (cudaMemsetAsync(w + h->L.rphys, 0, n_forward(D) * g.nreal * rb, h->stream) != cudaSuccess) return LBM_ERR_CUDA;
    if (cudaMemcpyAsync(w + h->L.rphys, d_phi, g.nreal * rb, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    if (d_u && cudaMemcpyAsync(w + h->L.rphys + g.nreal * rb, d_u, D * g.nreal * rb, cudaMemcpyDeviceToDevice,
                               h->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    const lbm_status s = h->params.precision == PFM_F64 ? exec<double>(h->fwd, false, w + h->L.rphys, w + h->L.cout)
                                                        : exec<float>(h->fwd, false, w + h->L.rphys, w + h->L.cout);
    if (s != LBM_OK) return s;
    if (cudaMemcpyAsync(w + h->L.phi_h, w + h->L.cout, g.ncplx * cb, cudaMemcpyDeviceToDevice, h->stream) !=
            cudaSuccess ||
        cudaMemcpyAsync(w + h->L.u_h, w + h->L.cout + g.ncplx * cb, D * g.ncplx * cb, cudaMemcpyDeviceToDevice,
                        h->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    h->started = 0;
    return LBM_OK;
}

LBM_SC_API lbm_status pfm_step(pfm_handle* h, int nsteps) {
    if (!h || nsteps < 0) return LBM_ERR_INVALID_ARG;
    if (nsteps > 0 && h->fused.ok) {
        return h->g.dim == 3 ? FusedRun<3>{h}.run(nsteps) : FusedRun<2>{h}.run(nsteps);
    }
    for (int i = 0; i < nsteps; ++i) {
        const lbm_status s = h->params.precision == PFM_F64 ? step_typed<double>(h) : step_typed<float>(h);
        if (s != LBM_OK) return s;
    }
    return LBM_OK;
}

LBM_SC_API lbm_status pfm_fields(pfm_handle* h, void* d_phi, void* d_u) {
    if (!h) return LBM_ERR_INVALID_ARG;
    const Geometry& g = h->g;
    const int D = g.dim;
    const size_t rb = real_bytes(&h->params);
    unsigned char* w = h->ws;
    lbm_status s;
    if (h->params.precision == PFM_F64) {
        pfm_prep_kernel<double><<<grid_for(g.ncplx), 256, 0, h->stream>>>(
            g, h->c, (const cufftDoubleComplex*)(w + h->L.phi_h), (const cufftDoubleComplex*)(w + h->L.u_h),
            (cufftDoubleComplex*)(w + h->L.cin));
        if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
        s = exec<double>(h->inv, true, w + h->L.cin, w + h->L.rin);
    } else {
        pfm_prep_kernel<float><<<grid_for(g.ncplx), 256, 0, h->stream>>>(
            g, h->c, (const cufftComplex*)(w + h->L.phi_h), (const cufftComplex*)(w + h->L.u_h),
            (cufftComplex*)(w + h->L.cin));
        if (cudaGetLastError() != cudaSuccess) return LBM_ERR_CUDA;
        s = exec<float>(h->inv, true, w + h->L.cin, w + h->L.rin);
    }
    if (s != LBM_OK) return s;
    if (d_phi && cudaMemcpyAsync(d_phi, w + h->L.rin, g.nreal * rb, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    if (d_u && cudaMemcpyAsync(d_u, w + h->L.rin + (size_t)(2 + D) * g.nreal * rb, D * g.nreal * rb,
                               cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess)
        return LBM_ERR_CUDA;
    return LBM_OK;
}

LBM_SC_API void pfm_destroy(pfm_handle* h) {
    if (!h) return;
    cufftDestroy(h->inv);
    cufftDestroy(h->fwd);
    delete h;
}

}  // extern "C"

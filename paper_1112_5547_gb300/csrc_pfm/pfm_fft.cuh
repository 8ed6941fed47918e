// The FP64 phase-field step with its transforms inside its own kernels.
//
// A step needs 2 + 2 D real fields in physical space and 2 + D + D (D + 1) / 2
// products back in Fourier space; in FP64 it is bound by the FP64 units (two FMA a
// clock and SM), so what counts is the number of operations.  One kernel per axis
// does everything that is local to a line of that axis:
//   spectral axis (z in 3D, y in 2D): forward transforms along it, S^, N^, the
//     AB2 / CN update, and the next step's inverse transforms along it;
//   y (3D): inverse; forward (two kernels, x lies between them);
//   x: inverse to real space, the nonlinear terms, forward again.
// Derivatives are multiplications by i k, so a derivative along an axis that is
// still in Fourier space is formed there and needs no transform of its own on
// the axes done before: phi, its derivative along the spectral axis, lap phi and u
// go in (3 + D fields), and outwards -i k_b (u_a u_b) joins F_a as soon as axis b is
// transformed (2 + 2 D fields arrive).  The element-wise passes between the
// transforms are gone, with their divisions.  GB300, ms a step with batched
// transforms and separate kernels, and so: 512^2 0.467 / 0.331, 128^3 4.83 / 3.27; small
// and narrow boxes are faster with batched transforms (fused_pays in pfm.cu).
// (The FP32 step is bound by memory and instruction issue instead: these kernels in
// FP32 took 2.8 ms at 256^3 against 2.2, so it keeps the batched transforms.)
//
// Transforms: Stockham autosort in shared memory, radix 4 first and last and any of
// 2, 3, 4, 5, 8 between, so a length is 16 times a product of those.  In the column
// kernels a thread owns rows j + q n / 4 of one column before and after, so the
// first and last radix run in registers straight from and to global memory.  An
// inverse transform is the forward one with real and imaginary parts exchanged
// before and after.  Real lines (x) go as half-length complex ones (even and odd
// samples as real and imaginary parts).
#pragma once

#include <cuda_runtime.h>

namespace pfm_fft {

using C = double2;
constexpr int R0 = 4;  // radix of the first and last pass: values a thread holds
constexpr int kMaxMid = 8;
struct Plan {
    int n, nmid;
    int mid[kMaxMid];
};

// n = 16 times a product of 2, 3, 4, 5, 8; false: not of that form.
inline bool make_plan(int n, Plan* p) {
    p->n = n;
    p->nmid = 0;
    if (n % (R0 * R0) != 0) return false;
    int m = n / (R0 * R0);
    static const int radix[5] = {8, 4, 2, 3, 5};
    for (int r : radix)
        while (m % r == 0) {
            if (p->nmid == kMaxMid) return false;
            p->mid[p->nmid++] = r;
            m /= r;
        }
    return m == 1;
}

__device__ __forceinline__ C add(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ C sub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ C mul(C a, C b) { return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ C mni(C a) { return C{a.y, -a.x}; }   // -i a
__device__ __forceinline__ C swp(C a) { return C{a.y, a.x}; }
__device__ __forceinline__ C cnj(C a) { return C{a.x, -a.y}; }

// Forward DFT of R values in place, natural order.
template <int R> __device__ __forceinline__ void dft(C (&v)[R]) {
    using T = double;
    if constexpr (R == 2) {
        const C a = v[0], b = v[1];
        v[0] = add(a, b);
        v[1] = sub(a, b);
    } else if constexpr (R == 3) {
        const C t = add(v[1], v[2]), d = sub(v[1], v[2]);
        const T s = (T)0.86602540378443864676;
        const C m{v[0].x - (T)0.5 * t.x, v[0].y - (T)0.5 * t.y}, e{s * d.y, -s * d.x};  // -i s d
        v[0] = add(v[0], t);
        v[1] = add(m, e);
        v[2] = sub(m, e);
    } else if constexpr (R == 4) {
        const C a = add(v[0], v[2]), b = sub(v[0], v[2]), c = add(v[1], v[3]), d = mni(sub(v[1], v[3]));
        v[0] = add(a, c);
        v[1] = add(b, d);
        v[2] = sub(a, c);
        v[3] = sub(b, d);
    } else if constexpr (R == 5) {
        const T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;
        const T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;
        const C t1 = add(v[1], v[4]), t2 = add(v[2], v[3]), t3 = sub(v[1], v[4]), t4 = sub(v[2], v[3]);
        const C a1{v[0].x + c1 * t1.x + c2 * t2.x, v[0].y + c1 * t1.y + c2 * t2.y};
        const C a2{v[0].x + c2 * t1.x + c1 * t2.x, v[0].y + c2 * t1.y + c1 * t2.y};
        const C b1 = mni(C{s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y});
        const C b2 = mni(C{s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y});
        v[0] = add(v[0], add(t1, t2));
        v[1] = add(a1, b1);
        v[2] = add(a2, b2);
        v[3] = sub(a2, b2);
        v[4] = sub(a1, b1);
    } else {
        static_assert(R == 8, "radix");
        C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft<4>(e);
        dft<4>(o);
        const T s = (T)0.70710678118654752440;
        o[1] = C{s * (o[1].x + o[1].y), s * (o[1].y - o[1].x)};
        o[2] = mni(o[2]);
        o[3] = C{s * (o[3].y - o[3].x), -s * (o[3].x + o[3].y)};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = add(e[k], o[k]);
            v[k + 4] = sub(e[k], o[k]);
        }
    }
}

// One radix-R pass of M columns (a power of two, fastest over the threads) of
// length n from src to dst, Ns the transformed length so far; element i of column
// x at i M + x; tw[t] = e^{-2 pi i t / n}.
template <int R>
__device__ __forceinline__ void pass_columns(const C* src, C* dst, int n, int M, int Ns, int tid, int nt, const C* tw) {
    const int nb = n / R, step = nb / Ns, lg = 31 - __clz(M);
    for (int q = tid; q < nb * M; q += nt) {
        const int x = q & (M - 1), j = q >> lg;
        const int jm = j % Ns;
        C v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) {
            v[k] = src[(j + k * nb) * M + x];
            if (k > 0) v[k] = mul(v[k], tw[jm * k * step]);
        }
        dft<R>(v);
        const int o = (j - jm) * R + jm;
#pragma unroll
        for (int k = 0; k < R; ++k) dst[(o + k * Ns) * M + x] = v[k];
    }
}

// All middle passes; returns the buffer that holds the result (a synced one).  Not
// inlined: the copies in the spectral kernel overran the instruction cache.
__device__ __noinline__ inline C* middle_columns(C* src, C* dst, const Plan& p, int M, int tid, int nt, const C* tw) {
    int Ns = R0;
#pragma unroll 1
    for (int m = 0; m < p.nmid; ++m) {
        const int r = p.mid[m];
        switch (r) {
            case 2: pass_columns<2>(src, dst, p.n, M, Ns, tid, nt, tw); break;
            case 3: pass_columns<3>(src, dst, p.n, M, Ns, tid, nt, tw); break;
            case 4: pass_columns<4>(src, dst, p.n, M, Ns, tid, nt, tw); break;
            case 5: pass_columns<5>(src, dst, p.n, M, Ns, tid, nt, tw); break;
            default: pass_columns<8>(src, dst, p.n, M, Ns, tid, nt, tw); break;
        }
        __syncthreads();
        C* const t = src;
        src = dst;
        dst = t;
        Ns *= r;
    }
    return src;
}

// Rows: line l at l pitch, element i at i + i / 16 (a shift of one value every 16
// spreads the strided writes over the banks); tw2[t] = e^{-2 pi i t / (2 n)}.  A thread
// keeps its butterfly j for all its lines, so the twiddles and the indices are
// formed once per pass.
__device__ __forceinline__ int pad16(int i) { return i + (i >> 4); }
template <class Body> __device__ __forceinline__ void for_rows(int nb, int lines, int tid, int nt, const Body& body) {
    const int per = nb < nt ? nb : nt, par = nt / per, l0 = tid / per;
    if (l0 >= par) return;
    for (int j = tid - l0 * per; j < nb; j += per) body(j, l0, par);
}
template <int R>
__device__ __forceinline__ void pass_rows(const C* src, C* dst, int n, int lines, int pitch, int Ns, int tid, int nt,
                                          const C* tw2, bool exchange = false) {
    const int nb = n / R, step = 2 * (nb / Ns);
    for_rows(nb, lines, tid, nt, [&](int j, int l0, int par) {
        const int jm = j % Ns, o = (j - jm) * R + jm;
        C t[R];
#pragma unroll
        for (int k = 1; k < R; ++k) t[k] = tw2[jm * k * step];
        for (int l = l0; l < lines; l += par) {
            const C* const a = src + l * pitch;
            C* const b = dst + l * pitch;
            C v[R];
#pragma unroll
            for (int k = 0; k < R; ++k) {
                v[k] = a[pad16(j + k * nb)];
                if (k > 0) v[k] = mul(v[k], t[k]);
            }
            dft<R>(v);
#pragma unroll
            for (int k = 0; k < R; ++k) b[pad16(o + k * Ns)] = exchange ? swp(v[k]) : v[k];
        }
    });
}
__device__ __noinline__ inline C* middle_rows(C* src, C* dst, const Plan& p, int lines, int pitch, int tid, int nt, const C* tw2) {
    int Ns = R0;
#pragma unroll 1
    for (int m = 0; m < p.nmid; ++m) {
        const int r = p.mid[m];
        switch (r) {
            case 2: pass_rows<2>(src, dst, p.n, lines, pitch, Ns, tid, nt, tw2); break;
            case 3: pass_rows<3>(src, dst, p.n, lines, pitch, Ns, tid, nt, tw2); break;
            case 4: pass_rows<4>(src, dst, p.n, lines, pitch, Ns, tid, nt, tw2); break;
            case 5: pass_rows<5>(src, dst, p.n, lines, pitch, Ns, tid, nt, tw2); break;
            default: pass_rows<8>(src, dst, p.n, lines, pitch, Ns, tid, nt, tw2); break;
        }
        __syncthreads();
        C* const t = src;
        src = dst;
        dst = t;
        Ns *= r;
    }
    return src;
}

// Twiddle table of one axis: tw[t] = e^{-2 pi i t / n}.
__global__ void twiddle_kernel(C* tw, int n) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(2.0 * (double)t / (double)n, &s, &c);
        tw[t] = C{c, -s};
    }
}

// Transforms of M neighbouring columns, one field after the other: the thread
// (x = tid % M, j = tid / M) holds rows j + q n / R0 in v before and after.  Two
// buffers of n M values; the next field starts in the one that was not read last,
// which every thread has left by then.
struct Columns {
    const Plan& p;
    const C* tw;
    C* a;
    C* b;
    int M, tid, nt, x, j;
    __device__ __forceinline__ Columns(const Plan& plan, const C* gtw, unsigned char* smem, int m) : p(plan), M(m) {
        tid = threadIdx.x;
        nt = blockDim.x;
        C* const s = reinterpret_cast<C*>(smem);
        a = s;
        b = s + p.n * M;
        C* const t = s + 2 * p.n * M;
        tw = t;
        x = tid % M;
        j = tid / M;
        for (int k = tid; k < p.n; k += nt) t[k] = gtw[k];
        __syncthreads();
    }
    __device__ __forceinline__ int row(int q) const { return j + q * (p.n / R0); }
    __device__ __forceinline__ void run(C (&v)[R0]) {
        dft<R0>(v);
#pragma unroll
        for (int q = 0; q < R0; ++q) a[(j * R0 + q) * M + x] = v[q];
        __syncthreads();
        C* const src = middle_columns(a, b, p, M, tid, nt, tw);
        C* const other = src == a ? b : a;
#pragma unroll
        for (int q = 0; q < R0; ++q) {
            v[q] = src[row(q) * M + x];
            if (q > 0) v[q] = mul(v[q], tw[j * q]);
        }
        dft<R0>(v);
        b = src;
        a = other;
    }
    __device__ __forceinline__ void run_inverse(C (&v)[R0]) {
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = swp(v[q]);
        run(v);
#pragma unroll
        for (int q = 0; q < R0; ++q) v[q] = swp(v[q]);
    }
};

inline size_t columns_smem(int n, int M) { return ((size_t)2 * n * M + n) * sizeof(C); }

}  // namespace pfm_fft

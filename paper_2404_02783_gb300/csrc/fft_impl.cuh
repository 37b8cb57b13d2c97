// 3D real FFT passes and the fused spectral operators of the PM step, templated on
// precision and transform size (included by fft_f32.cu and fft_f64.cu).
//
// Data flow of a 3D r2c transform of a real mesh R[x][y][z] (side n):
//   z_r2c : rows along z -> half spectrum T[kz][x][y]  (kz = 0..n/2; transposing store)
//   y_rows: rows along y (contiguous)                  -> T[kz][x][ky]
//   x_cols: columns along x (stride n)                 -> S[kz][kx][ky]
// and the inverse runs x_cols -> y_rows -> z_c2r.  Every pass reads and writes each
// element once: loads go straight from global memory into registers, the butterflies
// run in registers, shared memory carries only the exchanges between stages.
//
// Slab rows g = field n + x index the z passes; the half spectrum of slab row g and
// frequency kz sits at row ((g / C) (n/2 + 1) + kz) C + g % C with C = n, i.e. the
// layout [field][kz][x][y].
#pragma once

#include <math.h>

#include <algorithm>
#include <type_traits>

#include "dfloat.cuh"
#include "fft.cuh"
#include "internal.h"

namespace pm {

template <typename T> __device__ __forceinline__ cplx<T> tw_global(int k);
// The per-stage table (fft.cuh) of the length-L plan_e transform in global memory: a few KB
// read by every CTA, so it stays in L1 and the passes need no set-up of their own.
template <typename T> __device__ __forceinline__ const cplx<T>* tw_stages();
template <typename T, int L>
__device__ __forceinline__ TwGlobal<cplx<T>> tw_plan() {
    return TwGlobal<cplx<T>>{tw_stages<T>() + L};
}
cudaError_t set_smem_once(const void* fn, size_t bytes);

// The per-stage twiddle table of a length-L transform of eight elements a thread, into shared
// memory (the persistent and whole-plane middle passes).
template <typename T, int L>
__device__ __forceinline__ void load_stage_twiddles(cplx<T>* tw) {
    constexpr int TE = tw_stage_entries(L, 8);
    for (int k = threadIdx.x; k < TE; k += blockDim.x) {
        int Ns = radix_at(L, 1, 8), off = 0;  // stages with span Ns > 1, in order
        while (k >= off + (radix_at(L, Ns, 8) - 1) * Ns) {
            off += (radix_at(L, Ns, 8) - 1) * Ns;
            Ns *= radix_at(L, Ns, 8);
        }
        const int R = radix_at(L, Ns, 8);
        const int r = (k - off) / Ns + 1, jm = (k - off) % Ns;
        tw[k] = tw_global<T>(jm * r * (1024 / (Ns * R)));
    }
}

// a / d in the per-mode operators.  The division's own instruction sequence, with its check for
// operands out of range, is a good part of what the x pass issues a mode.  FP32: the quotient by
// the approximate reciprocal and one Newton-Raphson correction from its remainder, which leaves
// the rounding of the last operation: the correctly rounded quotient but for a few in a million,
// neighbours of it.  d in 2^-126 .. 2^126 (the approximate reciprocal of more is 0) and |a| above
// 2^-100, or 0 (the remainder is a's last bits); the operators' k^2, constraint denominators and
// numerators lie far inside.  FP64 divides are slower still: the reciprocal of d by the iteration
// for 1/d, r <- r + r (1 - d r), started from the FP32 reciprocal of d, which must be normal, and
// run twice (the relative error squares each time: ~2^-23, then ~2^-46, then below the FP64
// rounding), times a.  pm_div_mode_check and pm_div_mode_check_f32 compare both with the division.
template <typename T> __device__ __forceinline__ T div_mode(T a, T d) {
    const T r = __fdividef(1.0f, d), q = a * r;
    return fmaf(fmaf(-q, d, a), r, q);
}
template <> __device__ __forceinline__ double div_mode<double>(double a, double d) {
    double r = (double)__frcp_rn((float)d);
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    return a * r;
}

// Opts a kernel into more than 48 KB of dynamic shared memory once per device, so that
// launches (including those recorded into a CUDA graph) make no further attribute calls.
static inline cudaError_t set_smem(const void* fn, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return set_smem_once(fn, bytes);
}

// Launch shapes (compile time).
// z passes: YB rows of one x slab a CTA, so that the transposed side moves segments of YB
// complex values: 128 bytes at least in FP32.
template <typename T, int LOGN> struct ZShape {
    static constexpr int N = 1 << LOGN, M = N / 2, E = plan_e(M), Q = M / E, RS = row_stride(M);
    static constexpr int YB = (N == 32 || N == 128 || N == 256) ? 32 : 16;
    static constexpr int THREADS = YB * Q;
    // the registers of E complex values and their temporaries decide the residency
    static constexpr int MINB = (E == 32 ? 512 : 1024) / (sizeof(T) == 8 ? 2 : 1) / (THREADS < 64 ? 64 : THREADS);
    static constexpr size_t SMEM = sizeof(cplx<T>) * (size_t)YB * RS;
};
// y passes: RB rows a CTA.
template <typename T, int LOGN> struct YShape {
    static constexpr int N = 1 << LOGN, E = plan_e(N), Q = N / E, RS = row_stride(N);
    static constexpr int THREADS = 128, RB = THREADS / Q;
    static constexpr int MINB = (E == 32 ? 512 : 1024) / (sizeof(T) == 8 ? 2 : 1) / THREADS;
    static constexpr int MINB3 = (E == 32 ? 512 : E == 16 ? 768 : 1024) / (sizeof(T) == 8 ? 2 : 1) / THREADS;  // y grad3
    static constexpr size_t SMEM = sizeof(cplx<T>) * (size_t)RB * RS;
};
// x passes: CB columns of one plane a CTA, CTAs of 64 to 256 threads with several an SM.  Eight
// columns (64-byte row segments) beat sixteen where a thread holds 16 or 32 values: 340 against
// 457 us for the Newtonian pass at 512^3 and 43 against 48 us at 256^3 when they were compared (313
// and 41 now), since the wider CTA halves the CTAs an SM that overlap one another's loads; below
// that sixteen are better.
template <typename T, int LOGN> struct XShape {
    static constexpr int N = 1 << LOGN, E = plan_e(N), Q = N / E;
    static constexpr int CB = (sizeof(T) == 8) ? (E == 32 ? 4 : 8) : (E >= 16 ? 8 : 16);
    static constexpr int THREADS = CB * Q;
    static constexpr size_t COL = (size_t)(N + N / E) * CB;  // exchange slots
};

// Row of (slab row gl = field n + x, frequency kz) in the half spectra [field][kz][x][ky].
template <int M, int LOGN>
__device__ __forceinline__ size_t spec_row(int gl, int kz) {
    return ((size_t)((gl >> LOGN) * (M + 1) + kz) << LOGN) + (gl & ((1 << LOGN) - 1));
}

// =============================================================== z: r2c
// sub is subtracted from every input value as it is loaded: the mean of a density mesh (its
// zero mode, which no operator of the path uses), so that the transform's rounding scales
// with the fluctuations rather than with the mean (kz_max: planes beyond it are not written).  With sub = 1, v - 1 is exact for v in
// [0.5, 2^24] and below 0.5 within half the spacing of the values near 1 (2^-25 in FP32).
template <typename T, int LOGN>
__global__ void __launch_bounds__(ZShape<T, LOGN>::THREADS, ZShape<T, LOGN>::MINB)
    k_z_r2c(const T* in, cplx<T>* __restrict__ out, T sub, int kz_max) {
    typedef cplx<T> C;
    typedef ZShape<T, LOGN> S;
    constexpr int N = S::N, M = S::M, E = S::E, Q = S::Q, YB = S::YB, RS = S::RS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_next();
    wait_previous();
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x;
    const int y0 = blockIdx.x * YB;
    const int gl = blockIdx.y;
    const int b = row_of<Q>(tid), t = tid % Q;
    const C* row = reinterpret_cast<const C*>(in + ((size_t)gl * N + y0 + b) * N);
    C v[1][E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[0][m] = row[t + m * Q];
#pragma unroll
    for (int m = 0; m < E; ++m) {
        v[0][m].x -= sub;
        v[0][m].y -= sub;
    }
    C* z = buf + b * RS;
    WarpRowEx<C, E> ex{z};
    fft_regs<M, 1, false>(v, t, tw_plan<T, M>(), ex);
    ex.begin();  // the row's exchange has been read
#pragma unroll
    for (int m = 0; m < E; ++m) z[t + m * Q] = v[0][m];
    __syncthreads();
    // the real transform from the packed one, the pair (k, M - k) at a time:
    //   X_k = P + w^k O, X_{M-k} = conj(P - w^k O), P, O = (z_k +- z*_{M-k}) / 2 [* -i]
    const int bb = tid % YB, k0 = tid / YB;
    constexpr int TWS = 1024 / N;  // exp(-2 pi i k / N) = global table entry k TWS
    auto pair = [&](int k) {
        const C z1 = buf[bb * RS + k], z2 = cconj(buf[bb * RS + ((M - k) & (M - 1))]);
        const C P = cscale(cadd(z1, z2), T(0.5));
        const C O = cmul(cscale(cmul_mi<false>(csub(z1, z2)), T(0.5)), tw_global<T>(k * TWS));
        if (k <= kz_max) out[spec_row<M, LOGN>(gl, k) * N + y0 + bb] = cadd(P, O);
        if (2 * k != M && M - k <= kz_max) out[spec_row<M, LOGN>(gl, M - k) * N + y0 + bb] = cconj(csub(P, O));
    };
#pragma unroll
    for (int it = 0; it < E / 2; ++it) pair(k0 + it * Q);
    if (k0 == 0) pair(M / 2);
}

// =============================================================== z: c2r
template <typename T> struct Ptr3 {
    const cplx<T>* in[3];
    T* out[3];
    T* zero = nullptr;  // optional plain mesh, set to 0 by the component-0 CTAs
    int rows = 1;       // row r of out[j] at out[j] + r rows n
};

template <typename T, int LOGN>
__global__ void __launch_bounds__(ZShape<T, LOGN>::THREADS, ZShape<T, LOGN>::MINB)
    k_z_c2r(Ptr3<T> P, unsigned gradz_mask, T kf0, const double* __restrict__ kf_arr) {
    typedef cplx<T> C;
    typedef ZShape<T, LOGN> S;
    constexpr int N = S::N, M = S::M, E = S::E, Q = S::Q, YB = S::YB, RS = S::RS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_next();
    wait_previous();
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int tid = threadIdx.x;
    const int comp = blockIdx.z;
    const bool grad = (gradz_mask >> comp) & 1u;
    const int y0 = blockIdx.x * YB;
    const int gl = blockIdx.y;
    const T kf = kf_arr ? T(kf_arr[gl >> LOGN]) : kf0;
    const C* inp = comp == 0 ? P.in[0] : (comp == 1 ? P.in[1] : P.in[2]);
    T* pout = comp == 0 ? P.out[0] : (comp == 1 ? P.out[1] : P.out[2]);
    // Each thread loads the pairs (X_k, X_{M-k}) of its column -- all of its strided row
    // segments in flight together -- and forms in registers
    //   Y_k = s + i d, Y_{M-k} = conj(s) + i conj(d), s = X_k + X*_{M-k},
    //   d = (X_k - X*_{M-k}) exp(+2 pi i k / N),
    // the M-point sequence whose inverse transform interleaves the real output.
    const int bb = tid % YB, k0 = tid / YB;
    const C* col = inp + spec_row<M, LOGN>(gl, 0) * N + y0 + bb;
    constexpr size_t KZ = (size_t)N * N;  // elements from one kz to the next
    C X1[E / 2], X2[E / 2], Xm;
#pragma unroll
    for (int it = 0; it < E / 2; ++it) {
        X1[it] = col[(k0 + it * Q) * KZ];
        X2[it] = col[(M - k0 - it * Q) * KZ];
    }
    if (k0 == 0) Xm = col[(M / 2) * KZ];
    constexpr int TWS = 1024 / N;  // exp(-2 pi i k / N) = global table entry k TWS
    C* r = buf + bb * RS;          // the FFT exchanges reuse the rows afterwards
    auto pair = [&](int k, C a, C c) {
        if (grad) {  // (-i kz) X, Nyquist kz -> 0
            const T kza = kf * T(k), kzc = (k == 0) ? T(0) : kf * T(M - k);
            a = cmake<C>(a.y * kza, -a.x * kza);
            c = cmake<C>(c.y * kzc, -c.x * kzc);
        }
        if (k == 0) {
            a.y = T(0);
            c.y = T(0);
        }
        const C s = cadd(a, cconj(c));
        const C d = cmulc(csub(a, cconj(c)), tw_global<T>(k * TWS));
        r[k] = cmake<C>(s.x - d.y, s.y + d.x);
        if (k > 0 && 2 * k != M) r[M - k] = cmake<C>(s.x + d.y, d.x - s.y);
    };
#pragma unroll
    for (int it = 0; it < E / 2; ++it) pair(k0 + it * Q, X1[it], X2[it]);
    if (k0 == 0) pair(M / 2, Xm, Xm);
    __syncthreads();
    const int b = row_of<Q>(tid), t = tid % Q;
    C* z = buf + b * RS;
    C v[1][E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[0][m] = z[t + m * Q];
    WarpRowEx<C, E> ex{z};
    fft_regs<M, 1, true>(v, t, tw_plan<T, M>(), ex);
    C* orow = reinterpret_cast<C*>(pout + ((size_t)gl * N + y0 + b) * N * P.rows);
#pragma unroll
    for (int m = 0; m < E; ++m) orow[t + m * Q] = v[0][m];
    if (P.zero && comp == 0) {  // the same rows of the mesh the caller clears for its next use
        C* zrow = reinterpret_cast<C*>(P.zero + ((size_t)gl * N + y0 + b) * N);
#pragma unroll
        for (int m = 0; m < E; ++m) zrow[t + m * Q] = cmake<C>(T(0), T(0));
    }
}

// =============================================================== y: contiguous rows
// In place when in == out.  Each row is one warp's (or part of one), so no CTA barriers.
template <typename T, int LOGN, bool INV>
__global__ void __launch_bounds__(YShape<T, LOGN>::THREADS, YShape<T, LOGN>::MINB)
    k_y_rows(const cplx<T>* in, cplx<T>* out, int64_t nrows) {
    typedef cplx<T> C;
    typedef YShape<T, LOGN> S;
    constexpr int N = S::N, E = S::E, Q = S::Q;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_next();
    wait_previous();
    const int b = row_of<Q>(threadIdx.x), t = threadIdx.x % Q;
    const int64_t r = (int64_t)blockIdx.x * S::RB + b;
    const bool ok = r < nrows;
    C v[1][E];
    const C* irow = in + r * N;
    if (ok) {
#pragma unroll
        for (int m = 0; m < E; ++m) v[0][m] = irow[t + m * Q];
    }
    WarpRowEx<C, E> ex{reinterpret_cast<C*>(smem_raw) + b * S::RS};
    fft_regs<N, 1, INV>(v, t, tw_plan<T, N>(), ex);
    C* orow = out + r * N;
    if (ok) {
#pragma unroll
        for (int m = 0; m < E; ++m) orow[t + m * Q] = v[0][m];
    }
}

// A' = IFFT_y(A), B' = IFFT_y(B), C' = IFFT_y(-i ky A) (in place when Aout == A, Bout == B).
// The three transforms run one after the other in the same registers; A is read twice (the
// second time from L2) rather than held beside its transform, which would halve the warps.
template <typename T, int LOGN>
__global__ void __launch_bounds__(YShape<T, LOGN>::THREADS, YShape<T, LOGN>::MINB3)
    k_y_grad3(const cplx<T>* A, const cplx<T>* B, cplx<T>* Aout, cplx<T>* Bout, cplx<T>* __restrict__ Cout,
              int64_t nrows, T kf0, const double* __restrict__ kf_arr, int64_t rows_per_field) {
    typedef cplx<T> C;
    typedef YShape<T, LOGN> S;
    constexpr int N = S::N, E = S::E, Q = S::Q;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_next();
    wait_previous();
    const int b = row_of<Q>(threadIdx.x), t = threadIdx.x % Q;
    const int64_t r = (int64_t)blockIdx.x * S::RB + b;
    const bool ok = r < nrows;
    const T kf = (kf_arr && ok) ? T(kf_arr[r / rows_per_field]) : kf0;
    WarpRowEx<C, E> ex{reinterpret_cast<C*>(smem_raw) + b * S::RS};
    const int64_t o = r * N + t;
    C v[1][E];
    if (ok) {
#pragma unroll
        for (int m = 0; m < E; ++m) v[0][m] = A[o + m * Q];
    }
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int i = t + m * Q;
        const T ky = (2 * m == E && t == 0) ? T(0) : kf * T(2 * m < E ? i : i - N);
        v[0][m] = cmake<C>(v[0][m].y * ky, -v[0][m].x * ky);
    }
    fft_regs<N, 1, true>(v, t, tw_plan<T, N>(), ex);
    if (ok) {
#pragma unroll
        for (int m = 0; m < E; ++m) Cout[o + m * Q] = v[0][m];
#pragma unroll
        for (int m = 0; m < E; ++m) v[0][m] = A[o + m * Q];
    }
    fft_regs<N, 1, true>(v, t, tw_plan<T, N>(), ex);
    if (ok) {
        // a thread's own elements of A, which no other thread reads
#pragma unroll
        for (int m = 0; m < E; ++m) Aout[o + m * Q] = v[0][m];
        // Bout may alias B, never A
#pragma unroll
        for (int m = 0; m < E; ++m) v[0][m] = B[o + m * Q];
    }
    fft_regs<N, 1, true>(v, t, tw_plan<T, N>(), ex);
    if (ok) {
#pragma unroll
        for (int m = 0; m < E; ++m) Bout[o + m * Q] = v[0][m];
    }
}

// =============================================================== x: strided columns + spectral operators
// A hint that brings the 128-byte line holding p into L2 (no register, no wait).
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p)); }

// The linearised Poisson-gauge constraint on one mode in the working precision:
// Phi = (num delta + cc Phi_old) / (k^2 + base), cc = 0 at the first force evaluation.
template <typename T> struct GrOp {
    T kf2, num, base, cc;
    __device__ __forceinline__ GrOp(const SpecOp& op, T kf2T) {
        const T H = T(op.calH), om = T(op.omm_a);
        kf2 = kf2T;
        num = T(-1.5) * H * H * om;
        cc = op.first ? T(0) : T(3) * H * T(op.inv_dtau);
        base = T(3) * H * H + T(4.5) * H * H * om + cc;
    }
    __device__ __forceinline__ cplx<T> solve(cplx<T> delta, cplx<T> old, int n2) const {
        const T r = div_mode(T(1), kf2 * T(n2) + base);
        return cmake<cplx<T>>((num * delta.x + cc * old.x) * r, (num * delta.y + cc * old.y) * r);
    }
};

// The modes |n|^2 <= n_lo^2 of the constraint, solved and kept in FP64 in the island
// ((n_lo + 1) (2 n_lo + 1)^2 modes a field); the zero mode is 0.
template <typename T>
__device__ __noinline__ cplx<T> gr_island_mode(const SpecOp& op, cplx<T> vv, int nx, int ny, int nz, int n2, int field,
                                               double kf) {
    const int L = op.n_lo, W2 = 2 * L + 1;
    const size_t id = (((size_t)field * (L + 1) + nz) * W2 + (nx + L)) * W2 + (ny + L);
    if (n2 == 0) {
        if (L > 0) op.island[id] = make_double2(0.0, 0.0);
        return cmake<cplx<T>>(T(0), T(0));
    }
    const double k2 = kf * kf * (double)n2;
    const double H = op.calH;
    const double num_s = -1.5 * H * H * op.omm_a;
    double den = k2 + 3.0 * H * H + 4.5 * H * H * op.omm_a;
    double2 P = make_double2(num_s * (double)vv.x, num_s * (double)vv.y);
    if (!op.first) {
        const double2 old = op.island[id];
        const double cc = 3.0 * H * op.inv_dtau;
        P.x += cc * old.x;
        P.y += cc * old.y;
        den += cc;
    }
    P.x /= den;
    P.y /= den;
    op.island[id] = P;
    return cmake<cplx<T>>(T(P.x * op.ac2_over_n3), T(P.y * op.ac2_over_n3));
}

// The constraint on a thread's E modes kx = t + m Q of the x pass, in place (phi), Phi_old at
// old[i N].  The island's modes take the few columns near the origin out of line; the others'
// Phi_old are loaded eight at a time ahead of the arithmetic, since each store that follows
// keeps the next load from moving above it (one mode at a time made a chain of E L2 latencies).
template <typename T, int N, int E, int Q>
__device__ __forceinline__ void gr_modes(const SpecOp& op, cplx<T>* v, int t, int ny, int nz, int field, double kf,
                                         T kf2T, cplx<T>* old) {
    typedef cplx<T> C;
    const int nyz2 = ny * ny + nz * nz, nlo2 = op.n_lo * op.n_lo;
    const GrOp<T> g(op, kf2T);
    const T out = T(op.ac2_over_n3);
    if (nyz2 <= nlo2) {
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int nx = (2 * m < E) ? t + m * Q : t + m * Q - N;
            const int n2 = nx * nx + nyz2;
            if (n2 <= nlo2) v[m] = gr_island_mode<T>(op, v[m], nx, ny, nz, n2, field, kf);
        }
    }
    constexpr int G = E < 8 ? E : 8;
#pragma unroll
    for (int m0 = 0; m0 < E; m0 += G) {
        C o[G];
#pragma unroll
        for (int m = 0; m < G; ++m)
            o[m] = op.first ? cmake<C>(T(0), T(0)) : old[(size_t)(t + (m0 + m) * Q) * N];
#pragma unroll
        for (int m = m0; m < m0 + G; ++m) {
            const int nx = (2 * m < E) ? t + m * Q : t + m * Q - N;
            const int n2 = nx * nx + nyz2;
            if (n2 > nlo2) {
                const C P = g.solve(v[m], o[m - m0], n2);
                old[(size_t)(t + m * Q) * N] = P;
                v[m] = cscale(P, out);
            }
        }
    }
}

// The Zel'dovich filter (ZaFilter) on a thread's E modes kx = t + m Q of the x pass, in place:
// FP64 for the FP64 path; for FP32 the same value from pairs of FP32 numbers (an FP64 divide a mode
// made the pass 1.8 ms at 512^3), the amplitudes of eight modes loaded ahead of their use.
template <typename T, int N, int E, int Q>
__device__ __forceinline__ void za_modes(const SpecOp& op, cplx<T>* v, int t, int ny, int nz, int field, double kf) {
    typedef cplx<T> C;
    constexpr int M = N / 2, G = E < 8 ? E : 8;
    const int nyz2 = ny * ny + nz * nz;
    const bool nyq_yz = (2 * ny == -N) || (nz == M);
    const double c = op.za_filter == ZA_IDENTITY ? op.coef : op.coef / (kf * kf);
    const df cf = df_of(c);
    const int64_t tab = (int64_t)field * op.amp_stride;
#pragma unroll
    for (int m0 = 0; m0 < E; m0 += G) {
        typename std::conditional<sizeof(T) == 8, double, df>::type amp[G];
        if (op.za_filter == ZA_AMP) {
#pragma unroll
            for (int m = 0; m < G; ++m) {
                const int nx = (2 * (m0 + m) < E) ? t + (m0 + m) * Q : t + (m0 + m) * Q - N;
                if constexpr (sizeof(T) == 8) amp[m] = __ldg(static_cast<const double*>(op.amp) + tab + nx * nx + nyz2);
                else {
                    const float2 p = __ldg(static_cast<const float2*>(op.amp) + tab + nx * nx + nyz2);
                    amp[m] = df{p.x, p.y};
                }
            }
        }
#pragma unroll
        for (int m = m0; m < m0 + G; ++m) {
            const int nx = (2 * m < E) ? t + m * Q : t + m * Q - N;
            const int n2 = nx * nx + nyz2;
            C g = v[m];
            if (op.fixed_amp) {  // keep the phase, set |g| = 1
                const T r2 = g.x * g.x + g.y * g.y;
                g = (r2 > T(0)) ? cscale(g, rsqrt(r2)) : cmake<C>(T(0), T(0));
            }
            T filt;
            if (op.za_filter == ZA_IDENTITY) {
                filt = T(c);
            } else if constexpr (sizeof(T) == 8) {
                filt = (op.za_filter == ZA_AMP ? c * amp[m - m0] : c) / (double)n2;
            } else {
                filt = round_df(df_div(op.za_filter == ZA_AMP ? cf * amp[m - m0] : cf, (float)(n2 > 0 ? n2 : 1)));
            }
            v[m] = (n2 == 0 || nyq_yz || 2 * nx == -N) ? cmake<C>(T(0), T(0)) : cscale(g, filt);
        }
    }
}

// The per-mode operator of the x pass on mode (nx, ny, nz), |n|^2 = n2, of field `field`:
// the Newtonian Green's function (or the potential alone), or the linearised Poisson-gauge constraint (which reads and updates its Phi history at `old` and,
// for |n| <= n_lo, the FP64 island).  Returns phi for the mode.
template <typename T, int KIND, int N>
__device__ __forceinline__ cplx<T> mode_op(const SpecOp& op, cplx<T> vv, int nx, int ny, int nz, int n2, int field,
                                           double kf, T kfT, T coefT, T kf2T, cplx<T>* old) {
    typedef cplx<T> C;
    constexpr int M = N / 2;
    C phi;
    if constexpr (KIND == OP_NEWTON || KIND == OP_POTENTIAL) {
        phi = (n2 == 0) ? cmake<C>(T(0), T(0)) : cscale(vv, div_mode(coefT, T(n2)));
    } else {  // OP_GR
        if (n2 <= op.n_lo * op.n_lo) {
            phi = gr_island_mode<T>(op, vv, nx, ny, nz, n2, field, kf);
        } else {
            const C o = op.first ? cmake<C>(T(0), T(0)) : *old;
            const C Pc = GrOp<T>(op, kf2T).solve(vv, o, n2);
            *old = Pc;
            phi = cscale(Pc, T(op.ac2_over_n3));
        }
    }
    return phi;
}

// Registers of the x passes: kinds that hold a second sequence (phi beside its transform, or
// the second field of a cross spectrum) take twice the data registers.
template <typename T, int LOGN, int KIND> struct XRes {
    static constexpr bool TWO = KIND != OP_FWD_STORE && KIND != OP_INV && KIND != OP_POTENTIAL && KIND != OP_BIN;
    static constexpr int DATA = plan_e(1 << LOGN) * 2 * (int)sizeof(T) / 4 * (TWO ? 2 : 1);  // registers
    static constexpr int REGS = DATA <= 32 ? 64 : DATA <= 64 ? 104 : DATA <= 128 ? 168 : 255;
    static constexpr int MINB = 65536 / (REGS * XShape<T, LOGN>::THREADS);
};

// CTAs walk blocks blk = blockIdx.x, + gridDim.x, ... of CB columns of one plane (plane =
// blk / (N / CB)); several CTAs an SM overlap one another's loads, butterflies and stores.  The
// binning pass runs one CTA for each row of bin sums, the others one for each block.
template <typename T, int LOGN, int KIND>
__global__ void __launch_bounds__(XShape<T, LOGN>::THREADS, XRes<T, LOGN, KIND>::MINB)
    k_x_cols(cplx<T>* data, cplx<T>* __restrict__ out2, SpecOp op, int nplanes) {
    typedef cplx<T> C;
    typedef XShape<T, LOGN> S;
    constexpr int N = S::N, M = N / 2, E = S::E, Q = S::Q, CB = S::CB;
    constexpr int NCG = N / CB;  // column groups per plane
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_next();
    wait_previous();
    C* buf = reinterpret_cast<C*>(smem_raw);
    // OP_BIN: 1 / W^2 of the CIC window per |n_j| (W per axis from the FP64 table), in T
    T* iw2 = reinterpret_cast<T*>(buf + S::COL);
    constexpr bool BIN = KIND == OP_BIN || KIND == OP_BIN_CROSS, cross = KIND == OP_BIN_CROSS;
    const int tid = threadIdx.x;
    const int b = tid % CB, t = tid / CB;
    const int64_t nblk = (int64_t)nplanes * NCG;
    const auto tw = tw_plan<T, N>();
    CtaColEx<C, E, CB> ex{buf + b};
    if constexpr (BIN) {
        for (int e = tid; e <= M; e += S::THREADS) iw2[e] = op.deconv ? T(1.0 / (op.wtab[e] * op.wtab[e])) : T(1);
        __syncthreads();
    }
    // OP_BIN: this CTA's row of per-bin sums in global memory (zeroed by the caller); blockIdx.y
    // selects one of several fields, whose rows follow one another
    const size_t row = (size_t)blockIdx.y * op.acc_rows + blockIdx.x;
    double* acc_row = BIN ? op.acc + row * op.nbins : nullptr;
    if constexpr (BIN) data += (size_t)blockIdx.y * (M + 1) * N * N;
    // with a cross spectrum, optionally the auto spectrum of the second field in the same pass
    double* acc2_row = (cross && op.acc2) ? op.acc2 + row * op.nbins : nullptr;
#pragma unroll 1
    for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        const int plane = (int)(blk / NCG);
        const int kz = plane % (M + 1);
        const int field = plane / (M + 1);
        const double kf = op.kf_arr ? op.kf_arr[field] : op.kf;
        const int c = (int)(blk % NCG) * CB + b;
        const size_t pbase = (size_t)plane * N * N;
        if constexpr (BIN) {
            // every mode of the block beyond the last bin (a fifth of them with the whole sphere)
            const int c0 = c - b, ymin = c0 < M ? c0 : N - c0 - CB + 1;
            if (ymin * ymin + kz * kz > op.n2_max) continue;
        }
        C* base = data + pbase + c;
        C v[1][E];
#pragma unroll
        for (int m = 0; m < E; ++m) v[0][m] = base[(size_t)(t + m * Q) * N];
        if constexpr (KIND == OP_GR) {
            // the Poisson-gauge constraint reads the block's Phi_old after the forward transform:
            // its lines are brought into L2 beside the data
            constexpr int LINES = CB * (int)sizeof(C) >= 128 ? CB * (int)sizeof(C) / 128 : 1;
            const C* ph = reinterpret_cast<const C*>(op.phi_old) + pbase + (c - b);
            if (!op.first)
                for (int q = tid; q < N * LINES; q += S::THREADS)
                    prefetch_l2(reinterpret_cast<const char*>(ph + (size_t)(q / LINES) * N) + 128 * (q % LINES));
        }
        if (op.fwd) fft_regs<N, 1, false>(v, t, tw, ex);
        if constexpr (KIND == OP_FWD_STORE) {
#pragma unroll
            for (int m = 0; m < E; ++m) base[(size_t)(t + m * Q) * N] = v[0][m];
            continue;
        }
        if constexpr (KIND == OP_INV) {
            fft_regs<N, 1, true>(v, t, tw, ex);
#pragma unroll
            for (int m = 0; m < E; ++m) base[(size_t)(t + m * Q) * N] = v[0][m];
            continue;
        }
        const int ny = (c < M) ? c : c - N;
        const int nyz2 = ny * ny + kz * kz;
        if constexpr (BIN) {
            C u[1][cross ? E : 1];
            if constexpr (cross) {
                const C* in2 = reinterpret_cast<const C*>(op.in2) + pbase + c;
#pragma unroll
                for (int m = 0; m < E; ++m) u[0][m] = in2[(size_t)(t + m * Q) * N];
                fft_regs<N, 1, false>(u, t, tw, ex);
            }
            // regroup through the exchange buffer so that the thread holds kx = E t + m
            // (m = 0..E-1): neighbouring kx mostly share a |k| bin, so runs merge in registers
            auto regroup = [&](C* w) {
                __syncthreads();  // the buffer's last reads
#pragma unroll
                for (int m = 0; m < E; ++m) {
                    const int i = t + m * Q;
                    ex.col[(i + i / E) * CB] = w[m];
                }
                __syncthreads();
#pragma unroll
                for (int m = 0; m < E; ++m) w[m] = ex.put(t, m);
            };
            regroup(v[0]);
            if constexpr (cross) regroup(u[0]);
            // The thread's modes kx = E t .. E t + E - 1 lie on one side of the Nyquist index, so
            // |n|^2 is monotone over them, and a bin is a contiguous range of |n|^2: when the first
            // and the last mode of a group of eight fall in the same bin (neither the zero mode nor
            // beyond (n/2)^2), so do all eight, and two table lookups replace eight.  Consecutive
            // modes of a bin are summed in registers, at most eight of them in the working precision
            // before they join the run's FP64 total; each run is added once to the CTA's row (native
            // FP64 reduction in L2).
            int run_bin = -1;
            T run_sum = T(0), run_sum2 = T(0);
            double run_tot = 0.0, run_tot2 = 0.0;
            const T wyz = iw2[ny < 0 ? -ny : ny] * iw2[kz] * T((kz == 0 || kz == M) ? 1 : 2);
            constexpr int G = E < 8 ? E : 8;
#pragma unroll
            for (int g = 0; g < E; g += G) {
                const int ia = E * t + g, ib = ia + G - 1;
                const int nxa = (ia < M) ? ia : ia - N, nxb = (ib < M) ? ib : ib - N;
                const int n2a = nxa * nxa + nyz2, n2b = nxb * nxb + nyz2;
                int bin_all = -1;
                if (n2a > 0 && n2b > 0 && n2a <= op.n2_max && n2b <= op.n2_max) {
                    const int ba = op.bin_of[n2a], bb = op.bin_of[n2b];
                    if (ba == bb) bin_all = ba;
                } else if (n2a > op.n2_max && n2b > op.n2_max) {
                    continue;
                }
#pragma unroll
                for (int m = g; m < g + G; ++m) {
                    const int nx = nxa + (m - g);
                    const int n2 = nx * nx + nyz2;
                    if (n2 == 0 || n2 > op.n2_max) continue;
                    const int bin = (bin_all >= 0) ? bin_all : op.bin_of[n2];
                    if (bin < 0) continue;
                    const C vv = v[0][m], uu = u[0][cross ? m : 0];
                    // w |delta_n|^2 / W^2 (or the cross product), w = 1 on the kz = 0, n/2 planes, 2 elsewhere
                    const T wgt = iw2[nx < 0 ? -nx : nx] * wyz;
                    const T val = (cross ? vv.x * uu.x + vv.y * uu.y : vv.x * vv.x + vv.y * vv.y) * wgt;
                    const T val2 = acc2_row ? (uu.x * uu.x + uu.y * uu.y) * wgt : T(0);
                    if (bin != run_bin) {
                        if (run_bin >= 0) {
                            atomicAdd(acc_row + run_bin, run_tot + (double)run_sum);
                            if (acc2_row) atomicAdd(acc2_row + run_bin, run_tot2 + (double)run_sum2);
                        }
                        run_bin = bin;
                        run_tot = run_tot2 = 0.0;
                        run_sum = val;
                        run_sum2 = val2;
                    } else {
                        run_sum += val;
                        run_sum2 += val2;
                    }
                }
                if (g + G < E) {
                    run_tot += (double)run_sum;
                    run_sum = T(0);
                    if (acc2_row) {
                        run_tot2 += (double)run_sum2;
                        run_sum2 = T(0);
                    }
                }
            }
            if (run_bin >= 0) {
                atomicAdd(acc_row + run_bin, run_tot + (double)run_sum);
                if (acc2_row) atomicAdd(acc2_row + run_bin, run_tot2 + (double)run_sum2);
            }
            continue;
        } else {
            // ---- per-mode operator on modes (kx = t + m Q, ky = c, kz)
            // per-thread constants, formed once in the working precision (no FP64 work per mode in FP32)
            const T kfT = T(kf);
            const T coefT = T(op.coef) / (kfT * kfT);
            const T kf2T = T(kf * kf);
            if constexpr (KIND == OP_GR) {
                gr_modes<T, N, E, Q>(op, v[0], t, ny, kz, field, kf, kf2T,
                                     reinterpret_cast<C*>(op.phi_old) + pbase + c);
            } else if constexpr (KIND == OP_ZA) {
                za_modes<T, N, E, Q>(op, v[0], t, ny, kz, field, kf);
            } else {
#pragma unroll
                for (int m = 0; m < E; ++m) {
                    const int i = t + m * Q;
                    const int nx = (2 * m < E) ? i : i - N;
                    v[0][m] = mode_op<T, KIND, N>(op, v[0][m], nx, ny, kz, nx * nx + nyz2, field, kf, kfT, coefT, kf2T,
                                                  nullptr);
                }
            }
            if constexpr (KIND != OP_POTENTIAL) {
                C u[1][E];
#pragma unroll
                for (int m = 0; m < E; ++m) {
                    const int i = t + m * Q;
                    const T kx = (2 * m == E && t == 0) ? T(0) : kfT * T(2 * m < E ? i : i - N);
                    u[0][m] = cmake<C>(v[0][m].y * kx, -v[0][m].x * kx);  // -i kx phi
                }
                fft_regs<N, 1, true>(u, t, tw, ex);
                C* o2 = out2 + pbase + c;
#pragma unroll
                for (int m = 0; m < E; ++m) o2[(size_t)(t + m * Q) * N] = u[0][m];
            }
            fft_regs<N, 1, true>(v, t, tw, ex);
#pragma unroll
            for (int m = 0; m < E; ++m) base[(size_t)(t + m * Q) * N] = v[0][m];
        }
    }
}

// =============================================================== fused middle passes
// The three passes between the forward z and the inverse z transforms of a force
// evaluation -- forward y, x with the Green's function (or the Poisson-gauge constraint)
// and the x gradient, inverse y with the y gradient -- touch only one kz plane of the half
// spectrum each.  One persistent launch runs them plane by plane: a CTA takes items from a
// queue (item = one phase on a block of rows or columns of one plane) in rounds; round r
// holds the forward-y items of plane r, the x items of plane r - LAG and the inverse-y items
// of plane r - 2 LAG, so a plane's intermediate spectra are read back a few planes after they
// were written, from L2, and only the z pass's spectrum (read) and the three y-inverted
// spectra (written) go through HBM: 4 half spectra instead of 10.
// An item of the x phase waits for the plane's forward-y items to be done, an inverse-y item
// for its x items.  Every item waited on was handed out earlier, to a CTA that is running,
// so every wait ends; each wait still gives up after kMidSpinLimit polls (about a second),
// sets the error word and lets the CTA go on, so that a fault cannot hang the GPU.
struct MidSync {
    unsigned* queue;   // next item
    unsigned* done_y;  // [nplanes] finished forward-y items
    unsigned* done_x;  // [nplanes] finished x items
    unsigned* error;   // nonzero: a wait gave up
};
constexpr unsigned kMidSpinLimit = 1u << 23;

template <typename T, int LOGN, int THREADS_> struct MidShape {
    static constexpr int N = 1 << LOGN, M = N / 2, QN = N / 8;
    static constexpr int THREADS = THREADS_;
    static constexpr int RB = THREADS / QN;  // rows of a y item
    static constexpr int CB = THREADS / QN;  // columns of an x item
    static constexpr int ITEMS = N / RB;     // items of each phase per plane
    static constexpr int MINB = 1024 / THREADS;  // 64 registers a thread
    typedef RowLayout<N> LAY;
    // twiddles + the larger of the y exchange (two rows buffers of RB rows) and the x exchange
    // (two sequences of N x (CB + 1))
    static constexpr int XWORDS = 2 * N * (CB + 1), YWORDS = 2 * RB * LAY::RS;
    static constexpr size_t SMEM = sizeof(cplx<T>) * (N + (XWORDS > YWORDS ? XWORDS : YWORDS));
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Thread 0 waits until *cnt reaches target (bounded), then the CTA proceeds.
__device__ __forceinline__ void mid_wait(const unsigned* cnt, unsigned target, unsigned* error) {
    if (threadIdx.x == 0) {
        unsigned polls = 0;
        while (ld_acquire_u32(cnt) < target) {
            if (++polls > kMidSpinLimit || *(volatile unsigned*)error) {
                atomicExch(error, 1u);
                break;
            }
            __nanosleep(128);
        }
    }
    __syncthreads();
}

// lag: rounds between the phases of one plane, chosen by the launcher so that an item's
// dependencies were handed out more items earlier than there are CTAs in flight.
template <typename T, int LOGN, int KIND, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
    k_mid(cplx<T>* __restrict__ A, cplx<T>* __restrict__ B, cplx<T>* __restrict__ Cs, SpecOp op, int nplanes, int lag,
          MidSync sync) {
    typedef cplx<T> C;
    typedef MidShape<T, LOGN, THREADS> SH;
    constexpr int N = SH::N, M = SH::M, Q = SH::QN, RB = SH::RB, CB = SH::CB, ITEMS = SH::ITEMS;
    typedef typename SH::LAY LAY;
    constexpr int RS = LAY::RS, CS = CB + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tws = reinterpret_cast<C*>(smem_raw);
    const TwShared<C> tw{tws};
    C* buf = tws + N;
    __shared__ unsigned s_item;
    const int tid = threadIdx.x;
    load_stage_twiddles<T, N>(tws);
    const unsigned rounds = (unsigned)(nplanes + 2 * lag);
    const unsigned total = rounds * 3 * ITEMS;
#pragma unroll 1
    for (;;) {
        __syncthreads();  // the previous item's last reads of s_item and of the exchange buffers
        if (tid == 0) s_item = *(volatile unsigned*)sync.error ? total : atomicAdd(sync.queue, 1u);
        __syncthreads();
        const unsigned it = s_item;
        if (it >= total) break;
        const int r = (int)(it / (3 * ITEMS)), k = (int)(it % (3 * ITEMS));
        const int phase = k / ITEMS, blk = k % ITEMS;
        const int plane = r - phase * lag;
        if (plane < 0 || plane >= nplanes) continue;
        const size_t pbase = (size_t)plane * N * N;
        const int kz = plane % (M + 1);
        const int field = plane / (M + 1);
        const double kf = op.kf_arr ? op.kf_arr[field] : op.kf;
        const T kfT = T(kf);
        if (phase == 0) {
            // ---- forward y of rows x = blk RB .. + RB (in place in A)
            const int b = tid / Q, t = tid % Q;
            C* row = A + pbase + (size_t)(blk * RB + b) * N;
            C v[1][8];
#pragma unroll
            for (int m = 0; m < 8; ++m) v[0][m] = __ldcg(row + t + m * Q);
            RowEx<C, 1, true, LAY> ex{buf, RB, RS, b, 0};
            fft_regs<N, 1, false>(v, t, tw, ex);
#pragma unroll
            for (int m = 0; m < 8; ++m) row[t + m * Q] = v[0][m];
        } else if (phase == 1) {
            // ---- x pass of columns c = blk CB .. + CB: forward x, per-mode operator, phi and
            //      -i kx phi back along x (phi in place in A, -i kx phi to B)
            mid_wait(sync.done_y + plane, ITEMS, sync.error);
            const int b = tid % CB, t = tid / CB;
            const int c = blk * CB + b;
            C* base = A + pbase;
            C v[2][8];
#pragma unroll
            for (int m = 0; m < 8; ++m) v[0][m] = __ldcg(base + (size_t)(t + m * Q) * N + c);
            ColEx<C, N> ex{buf, CS, b};
            fft_regs<N, 1, false>(v, t, tw, ex);
            const int ny = (c < M) ? c : c - N;
            const T coefT = T(op.coef) / (kfT * kfT);
            const T kf2T = T(kf * kf);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int i = t + m * Q;
                const int nx = (i < M) ? i : i - N;
                const int n2 = nx * nx + ny * ny + kz * kz;
                const C phi = mode_op<T, KIND, N>(op, v[0][m], nx, ny, kz, n2, field, kf, kfT, coefT, kf2T,
                                                  reinterpret_cast<C*>(op.phi_old) + pbase + (size_t)i * N + c);
                v[0][m] = phi;
                const T kx = (2 * nx == -N) ? T(0) : kfT * T(nx);
                v[1][m] = cmake<C>(phi.y * kx, -phi.x * kx);  // -i kx phi
            }
            fft_regs<N, 2, true>(v, t, tw, ex);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                base[(size_t)(t + m * Q) * N + c] = v[0][m];
                B[pbase + (size_t)(t + m * Q) * N + c] = v[1][m];
            }
        } else {
            // ---- inverse y of rows x = blk RB .. + RB: A <- IFFT_y(A), C <- IFFT_y(-i ky A),
            //      B <- IFFT_y(B)
            mid_wait(sync.done_x + plane, ITEMS, sync.error);
            const int b = tid / Q, t = tid % Q;
            const size_t ro = pbase + (size_t)(blk * RB + b) * N;
            C v[2][8];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int i = t + m * Q;
                const C a = __ldcg(A + ro + i);
                v[0][m] = a;
                const int ny = (i < M) ? i : i - N;
                const T ky = (2 * ny == -N) ? T(0) : kfT * T(ny);
                v[1][m] = cmake<C>(a.y * ky, -a.x * ky);
            }
            RowEx<C, 2, false, LAY> ex{buf, RB, RS, b, 0};
            fft_regs<N, 2, true>(v, t, tw, ex);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                A[ro + t + m * Q] = v[0][m];
                Cs[ro + t + m * Q] = v[1][m];
            }
#pragma unroll
            for (int m = 0; m < 8; ++m) v[0][m] = __ldcg(B + ro + t + m * Q);
            RowEx<C, 1, false, LAY> ex1{buf, RB, RS, b, 0};
            fft_regs<N, 1, true>(v, t, tw, ex1);
#pragma unroll
            for (int m = 0; m < 8; ++m) B[ro + t + m * Q] = v[0][m];
        }
        if (phase < 2) {
            __syncthreads();  // every store of the item is made before it is counted
            if (tid == 0) {
                __threadfence();
                atomicAdd((phase == 0 ? sync.done_y : sync.done_x) + plane, 1u);
            }
        }
    }
}

// =============================================================== whole kz planes in shared memory
// On meshes of 64^3 and 128^3 one kz plane of the half spectrum (N^2 complex: 128 KB in FP32 at
// N = 128) fits in a CTA's shared memory.  k_plane runs the middle of a force evaluation on it:
// forward y (rows), forward x (columns) with the per-mode operator, then for each force
// component j the inverse x and inverse y transforms of -i k_j phi, written straight to that
// component's spectrum (x to GX, y to GY, z over A; the z pass then needs no z gradient).  HBM
// sees one read of the plane and three writes.  A row's or a column's transform uses its own
// slots of the plane as its exchange space; phi stays in registers between the components.
template <typename T, int LOGN> struct PlaneShape {
    static constexpr int N = 1 << LOGN, M = N / 2, Q = N / 8;
    static constexpr int THREADS = 8 * N;          // 64 sequences of N at a time
    static constexpr int SEQ = THREADS / Q;
    static constexpr int ROUNDS = N / SEQ;
    static constexpr int MINB = (THREADS >= 1024) ? 1 : 1024 / THREADS;  // 64 registers a thread
    static constexpr size_t SMEM = sizeof(cplx<T>) * ((size_t)N + (size_t)N * N);
    static_assert(ROUNDS >= 1 && SEQ * ROUNDS == N, "whole rounds of rows and columns");
};

template <typename T, int LOGN, int KIND>
__global__ void __launch_bounds__(PlaneShape<T, LOGN>::THREADS, PlaneShape<T, LOGN>::MINB)
    k_plane(cplx<T>* __restrict__ A, cplx<T>* __restrict__ GX, cplx<T>* __restrict__ GY, SpecOp op, int nplanes) {
    typedef cplx<T> C;
    typedef PlaneShape<T, LOGN> SH;
    constexpr int N = SH::N, M = SH::M, Q = SH::Q, SEQ = SH::SEQ, ROUNDS = SH::ROUNDS;
    typedef RowLayout<N> LAY;  // a permutation within each row's N slots
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tws = reinterpret_cast<C*>(smem_raw);
    const TwShared<C> tw{tws};
    C* P = tws + N;
    const int tid = threadIdx.x;
    load_stage_twiddles<T, N>(tws);
    launch_next();
    wait_previous();
#pragma unroll 1
    for (int plane = blockIdx.x; plane < nplanes; plane += gridDim.x) {
        const size_t pbase = (size_t)plane * N * N;
        const int kz = plane % (M + 1);
        const int field = plane / (M + 1);
        const double kf = op.kf_arr ? op.kf_arr[field] : op.kf;
        const T kfT = T(kf);
        __syncthreads();  // the previous plane's last reads of P and of the twiddles' set-up
        for (int e = tid; e < N * N; e += SH::THREADS) P[e] = __ldcs(A + pbase + e);
        __syncthreads();
        // ---- forward y of the N rows
#pragma unroll 1
        for (int r = 0; r < ROUNDS; ++r) {
            const int b = tid / Q, t = tid % Q;
            C* row = P + (size_t)(r * SEQ + b) * N;
            C v[1][8];
#pragma unroll
            for (int m = 0; m < 8; ++m) v[0][m] = row[t + m * Q];
            RowEx<C, 1, false, LAY> ex{P + (size_t)r * SEQ * N, SEQ, N, b, 0};
            fft_regs<N, 1, false>(v, t, tw, ex);
            __syncthreads();  // the row's last exchange has been read
#pragma unroll
            for (int m = 0; m < 8; ++m) row[t + m * Q] = v[0][m];
        }
        __syncthreads();
        // ---- forward x of the N columns and the per-mode operator: phi in registers
        C phi[ROUNDS][8];
        const T coefT = T(op.coef) / (kfT * kfT);
        const T kf2T = T(kf * kf);
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) {
            const int b = tid % SEQ, t = tid / SEQ;
            const int c = r * SEQ + b;
            C v[1][8];
#pragma unroll
            for (int m = 0; m < 8; ++m) v[0][m] = P[(size_t)(t + m * Q) * N + c];
            ColEx<C, N> ex{P + r * SEQ, N, b};
            fft_regs<N, 1, false>(v, t, tw, ex);
            const int ny = (c < M) ? c : c - N;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const int i = t + m * Q;
                const int nx = (i < M) ? i : i - N;
                const int n2 = nx * nx + ny * ny + kz * kz;
                phi[r][m] = mode_op<T, KIND, N>(op, v[0][m], nx, ny, kz, n2, field, kf, kfT, coefT, kf2T,
                                                reinterpret_cast<C*>(op.phi_old) + pbase + (size_t)i * N + c);
            }
        }
        // ---- each component: -i k_j phi back along x (columns), then along y (rows), to its spectrum
#pragma unroll 1
        for (int j = 0; j < 3; ++j) {
            C* out = (j == 0) ? GX : (j == 1 ? GY : A);
            __syncthreads();  // every read of P by the previous pass is done
#pragma unroll
            for (int r = 0; r < ROUNDS; ++r) {
                const int b = tid % SEQ, t = tid / SEQ;
                const int c = r * SEQ + b;
                const int ny = (c < M) ? c : c - N;
                const T ky = (2 * ny == -N) ? T(0) : kfT * T(ny);
                const T kzv = (kz == M) ? T(0) : kfT * T(kz);
                C v[1][8];
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int i = t + m * Q;
                    const int nx = (i < M) ? i : i - N;
                    const T kx = (2 * nx == -N) ? T(0) : kfT * T(nx);
                    const T kj = (j == 0) ? kx : (j == 1 ? ky : kzv);
                    v[0][m] = cmake<C>(phi[r][m].y * kj, -phi[r][m].x * kj);  // -i k_j phi
                }
                ColEx<C, N> ex{P + r * SEQ, N, b};
                fft_regs<N, 1, true>(v, t, tw, ex);
                __syncthreads();  // the column's last exchange has been read
#pragma unroll
                for (int m = 0; m < 8; ++m) P[(size_t)(t + m * Q) * N + c] = v[0][m];
            }
            __syncthreads();
#pragma unroll 1
            for (int r = 0; r < ROUNDS; ++r) {
                const int b = tid / Q, t = tid % Q;
                const C* row = P + (size_t)(r * SEQ + b) * N;
                C v[1][8];
#pragma unroll
                for (int m = 0; m < 8; ++m) v[0][m] = row[t + m * Q];
                RowEx<C, 1, false, LAY> ex{P + (size_t)r * SEQ * N, SEQ, N, b, 0};
                fft_regs<N, 1, true>(v, t, tw, ex);
                C* orow = out + pbase + (size_t)(r * SEQ + b) * N;
#pragma unroll
                for (int m = 0; m < 8; ++m) orow[t + m * Q] = v[0][m];
            }
        }
    }
}

// =============================================================== x: adjoint combine
// Transposed force chain on the x pass: the three y-transformed spectra of the deposited
// adjoint momenta V_j (fields j = 0, 1, 2 back to back, [kz][x][ky]) are transformed
// along x one after the other and accumulated as out = sum_j i k_j c(k) V_j,
// c = coef / (kf^2 |n|^2) (zero mode 0, k_j = 0 at its Nyquist index), then transformed
// back along x into out ([kz][x][ky], ready for the inverse y and z passes).  GR: the
// Poisson-gauge operator of AdjGrOp instead of c(k), with the carried spectrum gr.Z.  FD (the
// first-order gradient): V is one scalar field and W = FFT_x V, without the i k_j factors.
// Registers: the sum, the field and (AHEAD) the next one.
template <typename T, int LOGN> struct AdjRes {
    static constexpr int DATA = plan_e(1 << LOGN) * 2 * (int)sizeof(T) / 4;
    static constexpr int REGS = DATA <= 16 ? 96 : DATA <= 32 ? 160 : DATA <= 64 ? 168 : 255;
    static constexpr int MINB = 65536 / (REGS * XShape<T, LOGN>::THREADS);
};

template <typename T, int LOGN, bool GR, bool FD>
__global__ void __launch_bounds__(XShape<T, LOGN>::THREADS, AdjRes<T, LOGN>::MINB)
    k_x_adj(const cplx<T>* V, cplx<T>* out, double kf, double coef, float4* __restrict__ zero, int64_t nzero4,
            AdjGrOp gr) {
    typedef cplx<T> C;
    typedef XShape<T, LOGN> S;
    constexpr int N = S::N, M = N / 2, E = S::E, Q = S::Q, CB = S::CB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    launch_next();
    wait_previous();
    const int tid = threadIdx.x;
    const int b = tid % CB, t = tid / CB;
    const int kz = blockIdx.y;
    const int c = blockIdx.x * CB + b;
    const size_t pbase = (size_t)kz * N * N;
    const size_t field = (size_t)(M + 1) * N * N;
    const auto tw = tw_plan<T, N>();
    {  // side job: clear `zero` (a buffer the caller has finished with), grid-stride
        const int64_t nthr = (int64_t)gridDim.x * gridDim.y * blockDim.x;
        for (int64_t e = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + tid; e < nzero4; e += nthr)
            zero[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const T kfT = T(kf);
    const T coefT = T(coef) / (kfT * kfT);
    const int ny = (c < M) ? c : c - N;
    const T kyT = (2 * ny == -N) ? T(0) : kfT * T(ny);
    const T kzT = (kz == M) ? T(0) : kfT * T(kz);
    C acc[1][E];
    CtaColEx<C, E, CB> ex{reinterpret_cast<C*>(smem_raw) + b};
    // with 16 elements or fewer a thread, the next field is loaded while this one is transformed
    constexpr bool AHEAD = !FD && E * sizeof(C) <= 128;
    C v[1][E];
    const C* col = V + pbase + c;
    if constexpr (AHEAD) {
#pragma unroll
        for (int m = 0; m < E; ++m) v[0][m] = col[(size_t)(t + m * Q) * N];
    }
#pragma unroll 1
    for (int j = 0; j < (FD ? 1 : 3); ++j) {
        C nx[AHEAD ? E : 1];
        if constexpr (!AHEAD) {
#pragma unroll
            for (int m = 0; m < E; ++m) v[0][m] = col[j * field + (size_t)(t + m * Q) * N];
        }
        if constexpr (AHEAD) {
            if (j < 2) {
#pragma unroll
                for (int m = 0; m < E; ++m) nx[m] = col[(j + 1) * field + (size_t)(t + m * Q) * N];
            }
        }
        fft_regs<N, 1, false>(v, t, tw, ex);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int i = t + m * Q;
            const int nx = (2 * m < E) ? i : i - N;
            const T kj = FD ? T(1) : (j == 0) ? ((2 * nx == -N) ? T(0) : kfT * T(nx)) : (j == 1 ? kyT : kzT);
            const C a = j == 0 ? cmake<C>(T(0), T(0)) : acc[0][m];
            acc[0][m] = cmake<C>(a.x + kj * v[0][m].x, a.y + kj * v[0][m].y);
        }
        if constexpr (AHEAD) {
#pragma unroll
            for (int m = 0; m < E; ++m) v[0][m] = nx[m];
        }
    }
    if constexpr (GR) {
        // per-evaluation constants in the working precision; den and src / carry per mode
        const T kf2 = kfT * kfT, H = T(gr.H), H1 = T(gr.H1);
        const T base = T(3) * H * H + T(4.5) * H * H * T(gr.om) + T(gr.cc);
        const T base1 = T(3) * H1 * H1 + T(4.5) * H1 * H1 * T(gr.om1) + T(gr.cc1);
        const T num = T(-1.5) * H * H * T(gr.om), cc1 = T(gr.cc1), KA = T(gr.K_ac2_n3);
        C* Zc = reinterpret_cast<C*>(gr.Z) + pbase + c;
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int i = t + m * Q;
            const int nx = (2 * m < E) ? i : i - N;
            const int n2 = nx * nx + ny * ny + kz * kz;
            const T k2 = kf2 * T(n2);
            const T src = (n2 == 0) ? T(0) : div_mode(num, k2 + base);
            const T carry = (n2 == 0) ? T(0) : div_mode(cc1, k2 + base1);
            C* zi = Zc + (size_t)i * N;
            const C zo = *zi, a = acc[0][m];
            // K a c^2 W + carry Z, W = i acc (spectral gradient) or acc (first order)
            const C Z = FD ? cmake<C>(KA * a.x + carry * zo.x, KA * a.y + carry * zo.y)
                           : cmake<C>(-KA * a.y + carry * zo.x, KA * a.x + carry * zo.y);
            *zi = Z;
            acc[0][m] = cscale(Z, src);
        }
    } else {
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int i = t + m * Q;
            const int nx = (2 * m < E) ? i : i - N;
            const int n2 = nx * nx + ny * ny + kz * kz;
            const T cc = (n2 == 0) ? T(0) : div_mode(coefT, T(n2));
            const C a = acc[0][m];
            acc[0][m] = FD ? cscale(a, cc) : cmake<C>(-cc * a.y, cc * a.x);  // (i) c sum_j k_j V_j
        }
    }
    fft_regs<N, 1, true>(acc, t, tw, ex);
#pragma unroll
    for (int m = 0; m < E; ++m) out[pbase + (size_t)(t + m * Q) * N + c] = acc[0][m];
}

// =============================================================== launchers
// Passes whose launches overlap (launch_chained).  Not the FP64 ones of 64^3 and 128^3: blocks that are
// placed while others still run pile up on the SMs that are free first, and these passes are bound by
// each SM's few FP64 units (potential of a 64^3 mesh 53 us in order and 156 overlapping, 128^3 334
// and 383; first-order step 102 and 109, 648 and 698).  At 32^3 every block finds an SM of its own (43
// and 33 us), from 256^3 on there are many blocks for each (2576 and 2566).
template <typename T, int LOGN> constexpr bool kOverlap = sizeof(T) == 4 || LOGN <= 5 || LOGN >= 8;

template <typename T, int LOGN>
cudaError_t z_r2c_n(const T* in, cplx<T>* out, int rows, cudaStream_t st, double sub, int kz_max) {
    typedef ZShape<T, LOGN> S;
    cudaError_t e = set_smem((const void*)k_z_r2c<T, LOGN>, S::SMEM);
    if (e != cudaSuccess) return e;
    return launch_chained(k_z_r2c<T, LOGN>, dim3(S::N / S::YB, rows), S::THREADS, S::SMEM, st, kOverlap<T, LOGN>, in, out,
                          (T)sub, kz_max);
}

template <typename T, int LOGN>
cudaError_t z_c2r_n(const Ptr3<T>& P, int ncomp, int rows, unsigned mask, double kf, cudaStream_t st,
                    const double* kf_arr) {
    typedef ZShape<T, LOGN> S;
    cudaError_t e = set_smem((const void*)k_z_c2r<T, LOGN>, S::SMEM);
    if (e != cudaSuccess) return e;
    return launch_chained(k_z_c2r<T, LOGN>, dim3(S::N / S::YB, rows, ncomp), S::THREADS, S::SMEM, st, kOverlap<T, LOGN>, P,
                          mask, (T)kf, kf_arr);
}

template <typename T, int LOGN, bool INV>
cudaError_t y_rows_n(const cplx<T>* in, cplx<T>* out, int64_t nrows, cudaStream_t st) {
    typedef YShape<T, LOGN> S;
    cudaError_t e = set_smem((const void*)k_y_rows<T, LOGN, INV>, S::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t nblk = (nrows + S::RB - 1) / S::RB;
    return launch_chained(k_y_rows<T, LOGN, INV>, dim3((unsigned)nblk), S::THREADS, S::SMEM, st, kOverlap<T, LOGN>, in,
                          out, nrows);
}

template <typename T, int LOGN>
cudaError_t y_grad3_n(const cplx<T>* A, const cplx<T>* B, cplx<T>* Ao, cplx<T>* Bo, cplx<T>* Co, int64_t nrows, double kf,
                      cudaStream_t st, const double* kf_arr, int64_t rows_per_field) {
    typedef YShape<T, LOGN> S;
    cudaError_t e = set_smem((const void*)k_y_grad3<T, LOGN>, S::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t nblk = (nrows + S::RB - 1) / S::RB;
    return launch_chained(k_y_grad3<T, LOGN>, dim3((unsigned)nblk), S::THREADS, S::SMEM, st, kOverlap<T, LOGN>, A, B,
                          Ao, Bo, Co, nrows, (T)kf, kf_arr, rows_per_field);
}

template <typename T, int LOGN>
cudaError_t forward_zy_n(const T* in, cplx<T>* spec, int batch, cudaStream_t st, double sub, int kz_max) {
    constexpr int N = 1 << LOGN, M = N / 2;
    cudaError_t e = z_r2c_n<T, LOGN>(in, spec, N * batch, st, sub, kz_max);
    if (e != cudaSuccess) return e;
    // one field: its planes up to kz_max come first
    const int64_t planes = batch == 1 ? std::min(kz_max, M) + 1 : (int64_t)batch * (M + 1);
    return y_rows_n<T, LOGN, false>(spec, spec, planes * N, st);
}

// A (phi after the inverse x pass) and B (-i kx phi) in the full layout; scratch holds
// one half spectrum for IFFT_y(-i ky A).
template <typename T, int LOGN>
cudaError_t inverse_yz_grad_n(cplx<T>* A, cplx<T>* B, cplx<T>* scratch, T* const* out, int batch, double kf,
                              const double* kf_arr, cudaStream_t st, T* zero, int rows_out) {
    constexpr int N = 1 << LOGN, M = N / 2;
    const int64_t rows = (int64_t)batch * (M + 1) * N;
    cudaError_t e = y_grad3_n<T, LOGN>(A, B, A, B, scratch, rows, kf, st, kf_arr, (int64_t)(M + 1) * N);
    if (e != cudaSuccess) return e;
    Ptr3<T> P;
    P.in[0] = B;        // IFFT_y(-i kx phi)   -> g_x
    P.in[1] = scratch;  // IFFT_y(-i ky phi)   -> g_y
    P.in[2] = A;        // IFFT_y(phi), -i kz  -> g_z
    for (int j = 0; j < 3; ++j) P.out[j] = out[j];
    P.zero = zero;
    P.rows = rows_out;
    return z_c2r_n<T, LOGN>(P, 3, N * batch, 4u, kf, st, kf_arr);
}

template <typename T, int LOGN, int KIND>
cudaError_t x_cols_n(cplx<T>* data, cplx<T>* out2, int nplanes, const SpecOp& op, cudaStream_t st) {
    typedef XShape<T, LOGN> S;
    const size_t smem = sizeof(cplx<T>) * S::COL + (op.kind == OP_BIN ? sizeof(T) * (S::N / 2 + 1) : 0);
    const void* fn = (const void*)k_x_cols<T, LOGN, KIND>;
    cudaError_t e = set_smem(fn, smem);
    if (e != cudaSuccess) return e;
    int64_t grid = (int64_t)nplanes * (S::N / S::CB);
    if (op.kind == OP_BIN) {  // one row of bin sums per CTA
        int per_sm = 1;
        e = resident_ctas(fn, S::THREADS, smem, &per_sm);
        if (e != cudaSuccess) return e;
        grid = std::min<int64_t>(grid, std::min<int64_t>((int64_t)per_sm * num_sms(), op.acc_rows));
    }
    return launch_chained(k_x_cols<T, LOGN, KIND>, dim3((unsigned)grid, op.kind == OP_BIN ? op.bin_fields : 1), S::THREADS,
                          smem, st, kOverlap<T, LOGN>, data, out2, op, nplanes);
}

template <typename T, int LOGN, int THREADS>
cudaError_t middle_n(cplx<T>* A, cplx<T>* B, cplx<T>* Cs, int nplanes, const SpecOp& op, unsigned* sync_words,
                     cudaStream_t st) {
    typedef MidShape<T, LOGN, THREADS> SH;
    const void* fn = op.kind == OP_GR ? (const void*)k_mid<T, LOGN, OP_GR, THREADS>
                                      : (const void*)k_mid<T, LOGN, OP_NEWTON, THREADS>;
    cudaError_t e = set_smem(fn, SH::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 1;
    e = resident_ctas(fn, SH::THREADS, SH::SMEM, &per_sm);
    if (e != cudaSuccess) return e;
    // the queue and the counters start at zero; the error word after them stays set once set
    e = cudaMemsetAsync(sync_words, 0, sizeof(unsigned) * (4 + 2 * (size_t)nplanes), st);
    if (e != cudaSuccess) return e;
    MidSync sync{sync_words, sync_words + 4, sync_words + 4 + nplanes, sync_words + 4 + 2 * (size_t)nplanes};
    const int grid = per_sm * num_sms();
    const int lag = std::max(2, (grid + 3 * SH::ITEMS - 1) / (3 * SH::ITEMS) + 1);
    if (op.kind == OP_GR)
        k_mid<T, LOGN, OP_GR, THREADS><<<grid, SH::THREADS, SH::SMEM, st>>>(A, B, Cs, op, nplanes, lag, sync);
    else
        k_mid<T, LOGN, OP_NEWTON, THREADS><<<grid, SH::THREADS, SH::SMEM, st>>>(A, B, Cs, op, nplanes, lag, sync);
    return cudaGetLastError();
}

template <typename T, int LOGN>
cudaError_t middle_shape(cplx<T>* A, cplx<T>* B, cplx<T>* Cs, int nplanes, const SpecOp& op, unsigned* sync_words,
                         int threads, cudaStream_t st) {
    switch (threads) {
        case 256: return middle_n<T, LOGN, 256>(A, B, Cs, nplanes, op, sync_words, st);
        case 512: return middle_n<T, LOGN, 512>(A, B, Cs, nplanes, op, sync_words, st);
        case 1024: return middle_n<T, LOGN, 1024>(A, B, Cs, nplanes, op, sync_words, st);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T, int LOGN>
cudaError_t plane_n(cplx<T>* A, cplx<T>* GX, cplx<T>* GY, int nplanes, const SpecOp& op, cudaStream_t st) {
    typedef PlaneShape<T, LOGN> SH;
    const void* fn = op.kind == OP_GR ? (const void*)k_plane<T, LOGN, OP_GR> : (const void*)k_plane<T, LOGN, OP_NEWTON>;
    cudaError_t e = set_smem(fn, SH::SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 1;
    e = resident_ctas(fn, SH::THREADS, SH::SMEM, &per_sm);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<int64_t>((int64_t)per_sm * num_sms(), nplanes);
    if (op.kind == OP_GR)
        return launch_chained(k_plane<T, LOGN, OP_GR>, dim3(grid), SH::THREADS, SH::SMEM, st, kOverlap<T, LOGN>, A, GX,
                              GY, op, nplanes);
    return launch_chained(k_plane<T, LOGN, OP_NEWTON>, dim3(grid), SH::THREADS, SH::SMEM, st, kOverlap<T, LOGN>, A, GX,
                          GY, op, nplanes);
}

template <typename T, int LOGN, bool GR, bool FD>
cudaError_t x_adj_k(const cplx<T>* V, cplx<T>* out, double kf, double coef, float* zero, int64_t nzero, cudaStream_t st,
                    const AdjGrOp& gr) {
    typedef XShape<T, LOGN> S;
    const size_t smem = sizeof(cplx<T>) * S::COL;
    cudaError_t e = set_smem((const void*)k_x_adj<T, LOGN, GR, FD>, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_x_adj<T, LOGN, GR, FD>, dim3(S::N / S::CB, S::N / 2 + 1), S::THREADS, smem, st, kOverlap<T, LOGN>, V,
                          out, kf, coef, (float4*)zero, zero ? nzero / 4 : 0, gr);
}

template <typename T, int LOGN>
cudaError_t x_adj_n(const cplx<T>* V, cplx<T>* out, double kf, double coef, float* zero, int64_t nzero,
                    cudaStream_t st, const AdjGrOp* gr, bool fd) {
    if (nzero % 4 != 0 || (zero && (uintptr_t)zero % 16 != 0)) return cudaErrorInvalidValue;
    if (gr && !gr->Z) return cudaErrorInvalidValue;
    const AdjGrOp g = gr ? *gr : AdjGrOp();
    if (gr) return fd ? x_adj_k<T, LOGN, true, true>(V, out, kf, coef, zero, nzero, st, g)
                      : x_adj_k<T, LOGN, true, false>(V, out, kf, coef, zero, nzero, st, g);
    return fd ? x_adj_k<T, LOGN, false, true>(V, out, kf, coef, zero, nzero, st, g)
              : x_adj_k<T, LOGN, false, false>(V, out, kf, coef, zero, nzero, st, g);
}

template <typename T, int LOGN>
cudaError_t x_cols_kind(cplx<T>* data, cplx<T>* out2, int nplanes, const SpecOp& op, cudaStream_t st) {
    switch (op.kind) {
        case OP_FWD_STORE: return x_cols_n<T, LOGN, OP_FWD_STORE>(data, out2, nplanes, op, st);
        case OP_INV: return x_cols_n<T, LOGN, OP_INV>(data, out2, nplanes, op, st);
        case OP_NEWTON: return x_cols_n<T, LOGN, OP_NEWTON>(data, out2, nplanes, op, st);
        case OP_GR: return x_cols_n<T, LOGN, OP_GR>(data, out2, nplanes, op, st);
        case OP_ZA: return x_cols_n<T, LOGN, OP_ZA>(data, out2, nplanes, op, st);
        case OP_BIN:
            return op.in2 ? x_cols_n<T, LOGN, OP_BIN_CROSS>(data, out2, nplanes, op, st)
                          : x_cols_n<T, LOGN, OP_BIN>(data, out2, nplanes, op, st);
        case OP_POTENTIAL: return x_cols_n<T, LOGN, OP_POTENTIAL>(data, out2, nplanes, op, st);
        default: return cudaErrorInvalidValue;
    }
}

#define PM_DISPATCH_LOGN(n, CALL)      \
    switch (ilog2(n)) {                \
        case 4: { constexpr int LG = 4; return CALL; } \
        case 5: { constexpr int LG = 5; return CALL; } \
        case 6: { constexpr int LG = 6; return CALL; } \
        case 7: { constexpr int LG = 7; return CALL; } \
        case 8: { constexpr int LG = 8; return CALL; } \
        case 9: { constexpr int LG = 9; return CALL; } \
        case 10: { constexpr int LG = 10; return CALL; } \
        default: return cudaErrorInvalidValue; \
    }

template <typename T>
cudaError_t z_r2c(const T* in, cplx<T>* out, int n, int batch, cudaStream_t st, double sub) {
    PM_DISPATCH_LOGN(n, (z_r2c_n<T, LG>(in, out, n * batch, st, sub, n)))
}

template <typename T>
cudaError_t z_c2r(const cplx<T>* const* in, T* const* out, int ncomp, int n, int batch, unsigned gradz_mask,
                  double kf, cudaStream_t st, const double* kf_arr, T* zero, int rows) {
    Ptr3<T> P;
    P.rows = rows;
    for (int j = 0; j < 3; ++j) {
        P.in[j] = in[j < ncomp ? j : 0];
        P.out[j] = out[j < ncomp ? j : 0];
    }
    P.zero = zero;
    PM_DISPATCH_LOGN(n, (z_c2r_n<T, LG>(P, ncomp, n * batch, gradz_mask, kf, st, kf_arr)))
}

template <typename T, bool INV>
cudaError_t y_rows(cplx<T>* data, int64_t nrows, int n, cudaStream_t st) {
    PM_DISPATCH_LOGN(n, (y_rows_n<T, LG, INV>(data, data, nrows, st)))
}

template <typename T>
cudaError_t y_rows_grad3(cplx<T>* A, cplx<T>* B, cplx<T>* Cc, int64_t nrows, int n, double kf, cudaStream_t st,
                         const double* kf_arr, int64_t rows_per_field) {
    PM_DISPATCH_LOGN(n, (y_grad3_n<T, LG>(A, B, A, B, Cc, nrows, kf, st, kf_arr, rows_per_field)))
}

// The fused middle passes (forward y, x with op, inverse y with the y gradient) on meshes of
// 256^3 and up with CTAs of `threads` (256, 512 or 1024); cudaErrorNotSupported for other sizes
// (the caller runs the separate passes).
template <typename T>
cudaError_t fft_middle(cplx<T>* A, cplx<T>* B, cplx<T>* Cs, int nplanes, int n, const SpecOp& op, unsigned* sync_words,
                       int threads, cudaStream_t st) {
    if (op.kind != OP_NEWTON && op.kind != OP_GR) return cudaErrorInvalidValue;
    switch (ilog2(n)) {
        case 8: return middle_shape<T, 8>(A, B, Cs, nplanes, op, sync_words, threads, st);
        case 9: return middle_shape<T, 9>(A, B, Cs, nplanes, op, sync_words, threads, st);
        case 10: return middle_shape<T, 10>(A, B, Cs, nplanes, op, sync_words, threads, st);
        default: return cudaErrorNotSupported;
    }
}

// The middle passes on whole kz planes in shared memory (meshes of 64^3 and 128^3):
// GX, GY and A receive -i k_j phi transformed back along x and y (A in place); the z pass
// then runs without its z gradient.  cudaErrorNotSupported for other sizes.
template <typename T>
cudaError_t fft_plane(cplx<T>* A, cplx<T>* GX, cplx<T>* GY, int nplanes, int n, const SpecOp& op, cudaStream_t st) {
    if (op.kind != OP_NEWTON && op.kind != OP_GR) return cudaErrorInvalidValue;
    switch (ilog2(n)) {
        case 6: return plane_n<T, 6>(A, GX, GY, nplanes, op, st);
        case 7: return plane_n<T, 7>(A, GX, GY, nplanes, op, st);
        default: return cudaErrorNotSupported;
    }
}

template <typename T>
cudaError_t x_adj(const cplx<T>* V, cplx<T>* out, int n, double kf, double coef, cudaStream_t st, float* zero,
                  int64_t nzero, const AdjGrOp* gr, bool fd) {
    PM_DISPATCH_LOGN(n, (x_adj_n<T, LG>(V, out, kf, coef, zero, nzero, st, gr, fd)))
}

template <typename T>
cudaError_t forward_zy(const T* in, cplx<T>* spec, int n, int batch, cudaStream_t st, double sub, int kz_max) {
    PM_DISPATCH_LOGN(n, (forward_zy_n<T, LG>(in, spec, batch, st, sub, kz_max)))
}

template <typename T>
cudaError_t inverse_yz_grad(cplx<T>* A, cplx<T>* B, cplx<T>* scratch, T* const* out, int n, int batch, double kf,
                            cudaStream_t st, const double* kf_arr, T* zero, int rows) {
    PM_DISPATCH_LOGN(n, (inverse_yz_grad_n<T, LG>(A, B, scratch, out, batch, kf, kf_arr, st, zero, rows)))
}

template <typename T>
cudaError_t x_cols(cplx<T>* data, cplx<T>* out2, int nplanes, int n, const SpecOp& op, cudaStream_t st) {
    PM_DISPATCH_LOGN(n, (x_cols_kind<T, LG>(data, out2, nplanes, op, st)))
}

#define PM_INST(T)                                                                                     \
    template cudaError_t z_r2c<T>(const T*, cplx<T>*, int, int, cudaStream_t, double);                 \
    template cudaError_t z_c2r<T>(const cplx<T>* const*, T* const*, int, int, int, unsigned, double,  \
                                  cudaStream_t, const double*, T*, int);                               \
    template cudaError_t y_rows<T, false>(cplx<T>*, int64_t, int, cudaStream_t);                      \
    template cudaError_t y_rows<T, true>(cplx<T>*, int64_t, int, cudaStream_t);                       \
    template cudaError_t y_rows_grad3<T>(cplx<T>*, cplx<T>*, cplx<T>*, int64_t, int, double,           \
                                         cudaStream_t, const double*, int64_t);                        \
    template cudaError_t x_cols<T>(cplx<T>*, cplx<T>*, int, int, const SpecOp&, cudaStream_t);      \
    template cudaError_t forward_zy<T>(const T*, cplx<T>*, int, int, cudaStream_t, double, int);        \
    template cudaError_t x_adj<T>(const cplx<T>*, cplx<T>*, int, double, double, cudaStream_t, float*, \
                                  int64_t, const AdjGrOp*, bool);                                       \
    template cudaError_t inverse_yz_grad<T>(cplx<T>*, cplx<T>*, cplx<T>*, T* const*, int, int, double,   \
                                            cudaStream_t, const double*, T*, int);

}  // namespace pm

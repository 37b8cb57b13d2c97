// Register-resident FFT engine (Stockham autosort), compile-time length L and E elements a
// thread.
//
// A length-L sequence is owned by Q = L/E threads; thread t holds the E elements t + m Q
// (m = 0..E-1) in registers.  A stage of radix R <= E performs E/R butterflies per thread:
// butterfly j = t + q Q reads elements j + r L/R, multiplies by exp(-+2 pi i (j mod Ns) r /
// (Ns R)) and runs a register DFT of size R; the result element (j / Ns) Ns R + (j mod Ns) +
// r Ns goes through shared memory to whichever thread reads it in the next stage.  Loads of
// stage one and stores after the last stage touch elements t + m Q, i.e. consecutive threads
// touch consecutive elements, so callers stream them to and from global memory directly.
//
// plan_e picks E so that every length up to 1024 takes two stages, i.e. one exchange: an
// exchange costs 16 bytes of shared-memory traffic an element and a barrier, and the passes
// are bound by that pipe and by issue, not by registers.  The threads of a row then fit in one
// warp (Q <= 32) and its exchange needs only __syncwarp.  With eight elements a thread (three
// stages at 512, CTA barriers) the passes of a 512^3 force evaluation took 432 (forward z + y),
// 457 (x) and 1317 us (inverse y + z with the gradients); they take 320, 313 and 977 us, the
// first and the last at the copy bandwidth over the bytes they move (2.15 and 6.46 GB).
//
// Twiddles come from a per-stage table (tw_stage_offset; values from the host FP64 table
// exp(-2 pi i k / 1024), rounded once), in shared or global memory; INV conjugates them
// (unnormalised inverse).
#pragma once

#include "pm_common.cuh"

namespace pm {

// ---------------------------------------------------------------- butterflies
template <bool INV, typename C>
__device__ __forceinline__ void dft2(C& a, C& b) {
    C t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

// (x + iy) exp(-+ i pi/4) and (x + iy) exp(-+ 3 i pi/4), times sqrt 2.  The factor 1/sqrt 2 is
// left to the additions that follow, as one fused operation each (add_w8, sub_w8): the compiler does
// not contract the packed additions with a multiplication, and with the product rounded by itself
// the 512^3 transform was 2% further from 64 bits, its x pass took 325 us for 316, the inverse y and
// z passes 992 for 983.
template <bool INV, typename C>
__device__ __forceinline__ C rot_w8_1(C a) {
    return INV ? cmake<C>(a.x - a.y, a.x + a.y) : cmake<C>(a.x + a.y, a.y - a.x);
}
template <bool INV, typename C>
__device__ __forceinline__ C rot_w8_3(C a) {
    return INV ? cmake<C>(-a.x - a.y, a.x - a.y) : cmake<C>(a.y - a.x, -a.x - a.y);
}
// a + b, a - b, b times 1/sqrt 2 when W8
template <bool W8, typename C>
__device__ __forceinline__ C add_w8(C a, C b) {
    if constexpr (W8) return cfma(decltype(a.x)(0.70710678118654752440), b, a);
    else return cadd(a, b);
}
template <bool W8, typename C>
__device__ __forceinline__ C sub_w8(C a, C b) {
    if constexpr (W8) return cfma(decltype(a.x)(-0.70710678118654752440), b, a);
    else return csub(a, b);
}

// S2: v2 waits for its factor 1/sqrt 2, S13: v1 and v3 do.
template <bool INV, bool S2 = false, bool S13 = false, typename C>
__device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3) {
    C t0 = add_w8<S2>(v0, v2), t1 = sub_w8<S2>(v0, v2), t2 = cadd(v1, v3);
    C t3 = cmul_mi<INV>(csub(v1, v3));
    v0 = add_w8<S13>(t0, t2);
    v2 = sub_w8<S13>(t0, t2);
    v1 = add_w8<S13>(t1, t3);
    v3 = sub_w8<S13>(t1, t3);
}

// S4: v[4] waits for its factor 1/sqrt 2, S26: v[2] and v[6] do.
template <bool INV, bool S4 = false, bool S26 = false, typename C>
__device__ __forceinline__ void dft8(C* v) {
    // even / odd split: E = DFT4(v0 v2 v4 v6), O = DFT4(v1 v3 v5 v7); X_k = E_k + w^k O_k
    dft4<INV, S4, S26>(v[0], v[2], v[4], v[6]);
    dft4<INV>(v[1], v[3], v[5], v[7]);
    const C o1 = rot_w8_1<INV>(v[3]);
    const C o2 = cmul_mi<INV>(v[5]);
    const C o3 = rot_w8_3<INV>(v[7]);
    const C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = add_w8<true>(e1, o1); v[5] = sub_w8<true>(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = add_w8<true>(e3, o3); v[7] = sub_w8<true>(e3, o3);
}

// a exp(-+2 pi i J / 32), |J| <= 3, by three shears (the rotation of Paeth 1986): along x by
// tan(theta / 2), along y by sin(theta), along x again.  Three fused operations instead of two and
// two products, and the rounded constants are small beside 1: cos(pi/16) and cos(pi/8) are both
// nearly half a unit low in FP32.  Relative error of the r2c transform of white noise with cos and
// sin, and now: 1.61e-7 and 1.56e-7 (128^3), 1.77e-7 and 1.64e-7 (256^3), 1.93e-7 and 1.74e-7
// (512^3).  FP64 at 256^3, us: forward 863 -> 844, x 1331 -> 1293, inverse 2596 -> 2539.
template <int J, bool INV, typename C>
__device__ __forceinline__ C shear_w32(C a) {
    typedef decltype(a.x) T;
    constexpr int j = J < 0 ? -J : J;
    constexpr double tan_half = j == 1 ? 0.098491403357164253077 : j == 2 ? 0.19891236737965800691 : 0.30334668360734239168;
    constexpr double sine = j == 1 ? 0.19509032201612826785 : j == 2 ? 0.38268343236508977173 : 0.55557023301960222474;
    constexpr T sign = T((J < 0) != INV ? -1 : 1);
    constexpr T t = sign * T(tan_half), s = sign * T(sine);
    const T x = fma(t, a.y, a.x), y = fma(-s, x, a.y);
    return cmake<C>(fma(t, y, x), y);
}

// a exp(-+2 pi i J / 32), J = 0..31, times sqrt 2 for J = 4, 12, 20, 28
template <int J, bool INV, typename C>
__device__ __forceinline__ C mul_w32(C a) {
    if constexpr (J >= 16) {
        const C b = mul_w32<J - 16, INV>(a);
        return cmake<C>(-b.x, -b.y);
    } else if constexpr (J == 0) {
        return a;
    } else if constexpr (J == 4) {
        return rot_w8_1<INV>(a);
    } else if constexpr (J == 12) {
        return rot_w8_3<INV>(a);
    } else if constexpr (J == 8) {
        return cmul_mi<INV>(a);
    } else if constexpr (J < 4) {
        return shear_w32<J, INV>(a);
    } else if constexpr (J < 12) {
        return shear_w32<J - 8, INV>(cmul_mi<INV>(a));
    } else {
        const C b = shear_w32<J - 16, INV>(a);
        return cmake<C>(-b.x, -b.y);
    }
}

// A DFT of size 4 R2 as 4 x R2: DFT4 over the stride-R2 elements, the twiddles
// exp(-+2 pi i n2 k1 / (4 R2)), then DFT_R2 over n2 for each k1; X_{k1 + 4 k2}.  The eighth roots
// among the twiddles are those of n2 = R2 / 2 at k1 = 1, 3 and of n2 = R2 / 4, 3 R2 / 4 at k1 = 2:
// the elements whose factor the DFT_R2 takes into its first additions.
template <int R2, int N2, int K1, bool INV, typename C>
__device__ __forceinline__ void dft4xr_twiddle(C* v) {
    if constexpr (K1 < 4) {
        v[N2 + R2 * K1] = mul_w32<(N2 * K1 * (8 / R2)) % 32, INV>(v[N2 + R2 * K1]);
        dft4xr_twiddle<R2, N2, K1 + 1, INV>(v);
    } else if constexpr (N2 + 1 < R2) {
        dft4xr_twiddle<R2, N2 + 1, 1, INV>(v);
    }
}

template <int R2, bool INV, typename C>
__device__ __forceinline__ void dft4xr(C* v) {
    static_assert(R2 == 4 || R2 == 8, "DFT_R2 below");
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) dft4<INV>(v[n2], v[n2 + R2], v[n2 + 2 * R2], v[n2 + 3 * R2]);
    dft4xr_twiddle<R2, 1, 1, INV>(v);
    if constexpr (R2 == 8) {
        dft8<INV>(v);
        dft8<INV, true, false>(v + 8);
        dft8<INV, false, true>(v + 16);
        dft8<INV, true, false>(v + 24);
    } else {
        dft4<INV>(v[0], v[1], v[2], v[3]);
        dft4<INV, true, false>(v[4], v[5], v[6], v[7]);
        dft4<INV, false, true>(v[8], v[9], v[10], v[11]);
        dft4<INV, true, false>(v[12], v[13], v[14], v[15]);
    }
    C w[4 * R2];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) w[k1 + 4 * k2] = v[R2 * k1 + k2];
#pragma unroll
    for (int k = 0; k < 4 * R2; ++k) v[k] = w[k];
}

template <int R, bool INV, typename C>
__device__ __forceinline__ void dftR(C* v) {
    if constexpr (R == 32) dft4xr<8, INV>(v);
    else if constexpr (R == 16) dft4xr<4, INV>(v);
    else if constexpr (R == 8) dft8<INV>(v);
    else if constexpr (R == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 2) dft2<INV>(v[0], v[1]);
}

// Elements a thread of the row and column passes.
__host__ __device__ constexpr int plan_e(int L) { return L >= 512 ? 32 : L >= 128 ? 16 : L == 16 ? 4 : 8; }

__host__ __device__ constexpr int radix_at(int L, int Ns, int E) { return (L / Ns) >= E ? E : (L / Ns); }
__host__ __device__ constexpr int last_radix(int L, int E, int Ns = 1) {
    return (Ns * radix_at(L, Ns, E) >= L) ? radix_at(L, Ns, E) : last_radix(L, E, Ns * radix_at(L, Ns, E));
}

// Per-stage twiddle table: the stage with span Ns > 1 and radix R keeps
// w(r, jm) = exp(-2 pi i jm r / (Ns R)) at [offset(Ns) + (r - 1) Ns + jm], r = 1..R-1,
// jm = 0..Ns-1, so the lanes of a warp (consecutive jm) read consecutive entries.  The
// table of a length-L transform holds L - radix_at(L, 1, E) < L entries.
__host__ __device__ constexpr int tw_stage_offset(int L, int E, int Ns, int s = 1, int off = 0) {
    return (s >= Ns) ? off
                     : tw_stage_offset(L, E, Ns, s * radix_at(L, s, E), off + (s > 1 ? (radix_at(L, s, E) - 1) * s : 0));
}
__host__ __device__ constexpr int tw_stage_entries(int L, int E) { return tw_stage_offset(L, E, L); }

// Reads of the table: from shared memory, or (the plan_e transforms) from the global one.
template <typename C>
struct TwShared {
    const C* p;
    __device__ __forceinline__ C operator[](int e) const { return p[e]; }
};
template <typename C>
struct TwGlobal {
    const C* p;
    __device__ __forceinline__ C operator[](int e) const { return __ldg(p + e); }
};

// ---------------------------------------------------------------- exchangers
// Shared-memory rows of the exchanges of the whole-plane and persistent middle passes (rows of 64
// to 1024 elements): element i of a row sits at slot i ^ ((i >> 3) & MK) (a permutation within
// aligned blocks of MK + 1 elements), rows RS slots apart.  Chosen by enumerating every access
// pattern of a warp so that the 8-byte accesses of each half-warp fall in distinct banks.
template <int L>
struct RowLayout {
    static_assert(L >= 64 && L <= 1024, "lengths of the middle passes");
    static constexpr int MK = L >= 128 ? 15 : 7;
    static constexpr int RS = L >= 128 ? L + 1 : 72;
    __host__ __device__ static constexpr int slot(int i) { return i ^ ((i >> 3) & MK); }
};

// Rows: sequence s of row b at base[((p NSEQ + s) RB + b) RS + slot(i)]; two
// buffers alternate (p) when PP, so one barrier per exchange suffices.
template <typename C, int NSEQ, bool PP, class LAY>
struct RowEx {
    static constexpr bool kTwoStage = false;
    C* base;
    int RB, RS, b, p;
    __device__ __forceinline__ C& at(int s, int i) {
        return base[(((PP ? p : 0) * NSEQ + s) * RB + b) * RS + LAY::slot(i)];
    }
    __device__ __forceinline__ void begin() {
        if (!PP) __syncthreads();
    }
    __device__ __forceinline__ void sync() { __syncthreads(); }
    __device__ __forceinline__ void end() {
        if (PP) p ^= 1;
    }
};

// Columns: element i of column b of sequence s at base[(s L + i) CS + b] (columns
// interleaved so that lanes of consecutive columns hit consecutive banks).
template <typename C, int L>
struct ColEx {
    static constexpr bool kTwoStage = false;
    C* base;
    int CS, b;
    __device__ __forceinline__ C& at(int s, int i) { return base[(s * L + i) * CS + b]; }
    __device__ __forceinline__ void begin() { __syncthreads(); }
    __device__ __forceinline__ void sync() { __syncthreads(); }
    __device__ __forceinline__ void end() {}
};

// The plan_e transforms: element i of a sequence at slot i + i / E.  A writing thread holds E
// consecutive elements and a reading one elements Q apart, so with one spare slot every E both
// sides' lanes fall in distinct banks (E + 1 is odd).
//
// A row of Q <= 32 threads of one warp: only the warp synchronises.  Rows are row_stride slots
// apart (1 modulo 16), and row_of spaces the rows of a half-warp Q apart, so that rows sharing a
// half-warp use disjoint banks and a column of the rows can be walked without conflicts.
__host__ __device__ constexpr int row_stride(int L) { return (L + L / plan_e(L) + 14) / 16 * 16 + 1; }
template <int Q>
__device__ __forceinline__ int row_of(int tid) {
    if constexpr (Q == 32) return tid >> 5;
    const int g = (tid & 31) / Q;                 // group of Q lanes in the warp
    const int hg = g / (16 / (Q < 16 ? Q : 16));  // its half-warp
    const int gi = g % (16 / (Q < 16 ? Q : 16));
    const int idx = 2 * (tid >> 5) + hg;
    return (idx / Q) * 16 + gi * Q + idx % Q;
}
template <typename C, int E>
struct WarpRowEx {
    static constexpr bool kTwoStage = true;
    C* row;
    // the two sides of the exchange: result r of thread t (element t E + r), and element
    // j + r E of the reading butterfly j < E
    __device__ __forceinline__ C& put(int t, int r) { return row[t * (E + 1) + r]; }
    __device__ __forceinline__ C& get(int j, int r) { return row[j + r * (E + 1)]; }
    __device__ __forceinline__ void begin() { __syncwarp(); }
    __device__ __forceinline__ void sync() { __syncwarp(); }
    __device__ __forceinline__ void end() {}
};

// Columns of a CTA, interleaved: slot s of column b at s CB + b.
template <typename C, int E, int CB>
struct CtaColEx {
    static constexpr bool kTwoStage = true;
    C* col;  // the CTA's buffer + column b
    __device__ __forceinline__ C& put(int t, int r) { return col[(t * (E + 1) + r) * CB]; }
    __device__ __forceinline__ C& get(int j, int r) { return col[(j + r * (E + 1)) * CB]; }
    __device__ __forceinline__ void begin() { __syncthreads(); }
    __device__ __forceinline__ void sync() { __syncthreads(); }
    __device__ __forceinline__ void end() {}
};

// ---------------------------------------------------------------- stages
template <int L, int E, int Ns, int NSEQ, bool INV, typename C, class TW, class X>
__device__ __forceinline__ void fft_stages(C (*v)[E], int t, const TW& tw, X& ex) {
    constexpr int R = radix_at(L, Ns, E);
    constexpr int NB = E / R;
    constexpr int Q = L / E;
#pragma unroll
    for (int s = 0; s < NSEQ; ++s)
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            if constexpr (Ns > 1) {
                const int e0 = tw_stage_offset(L, E, Ns) + ((t + q * Q) & (Ns - 1));
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const C w = tw[e0 + (r - 1) * Ns];
                    v[s][q * R + r] = INV ? cmulc(v[s][q * R + r], w) : cmul(v[s][q * R + r], w);
                }
            }
            dftR<R, INV>(&v[s][q * R]);
        }
    if constexpr (Ns * R < L) {
        constexpr int Ns2 = Ns * R;
        constexpr int R2 = radix_at(L, Ns2, E);
        constexpr int NB2 = E / R2;
        ex.begin();
        if constexpr (X::kTwoStage) {
            // two stages, one sequence at a time
            static_assert(NSEQ == 1 && Ns == 1 && R == E && R2 == Q, "a plan_e transform takes two stages");
#pragma unroll
            for (int r = 0; r < R; ++r) ex.put(t, r) = v[0][r];
            ex.sync();
#pragma unroll
            for (int q = 0; q < NB2; ++q)
#pragma unroll
                for (int r = 0; r < R2; ++r) v[0][q * R2 + r] = ex.get(t + q * Q, r);
            ex.end();
            fft_stages<L, E, Ns2, NSEQ, INV>(v, t, tw, ex);
            return;
        } else {
#pragma unroll
            for (int s = 0; s < NSEQ; ++s)
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const int j = t + q * Q;
                    const int base = (j / Ns) * Ns2 + (j & (Ns - 1));
#pragma unroll
                    for (int r = 0; r < R; ++r) ex.at(s, base + r * Ns) = v[s][q * R + r];
                }
            ex.sync();
#pragma unroll
            for (int s = 0; s < NSEQ; ++s)
#pragma unroll
                for (int q = 0; q < NB2; ++q) {
                    const int j = t + q * Q;
#pragma unroll
                    for (int r = 0; r < R2; ++r) v[s][q * R2 + r] = ex.at(s, j + r * (L / R2));
                }
            ex.end();
            fft_stages<L, E, Ns2, NSEQ, INV>(v, t, tw, ex);
        }
    }
}

// Transform NSEQ sequences of length L (8 <= L <= 1024, a power of two), E elements a thread.
// On entry v[s][m] is element t + m L/E of sequence s; on exit v[s][m] is transform element
// t + m L/E.  Contains the exchanger's barriers: every thread of the CTA (or warp) must call it.
template <int L, int NSEQ, bool INV, int E, typename C, class TW, class X>
__device__ __forceinline__ void fft_regs(C (*v)[E], int t, const TW& tw, X& ex) {
    fft_stages<L, E, 1, NSEQ, INV>(v, t, tw, ex);
    constexpr int RL = last_radix(L, E);
    if constexpr (RL < E) {
        // after a closing radix-RL stage, slot q RL + r holds element t + (q + r E/RL) L/E
        constexpr int NB = E / RL;
#pragma unroll
        for (int s = 0; s < NSEQ; ++s) {
            C w[E];
#pragma unroll
            for (int q = 0; q < NB; ++q)
#pragma unroll
                for (int r = 0; r < RL; ++r) w[q + r * NB] = v[s][q * RL + r];
#pragma unroll
            for (int m = 0; m < E; ++m) v[s][m] = w[m];
        }
    }
}

}  // namespace pm

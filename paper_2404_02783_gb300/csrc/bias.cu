// Halo proxy for the linear-bias measurement (Sec. 5.2, Eq. b1): the ceil(f n^3)
// densest cells of a density mesh, ties broken by the lower linear index, turned into
// a tracer contrast delta_h = n_h / mean(n_h) - 1.
//
// Selection is exact: values map to order-preserving unsigned keys (sign-flip of the
// IEEE bits), a radix select finds the threshold key eleven bits at a time from the top
// (histograms of the cells that still match the chosen prefix), and of the cells equal to the
// threshold the lowest-index ones fill the remaining places.  The digits are chosen on the
// device, so nothing waits for the host between the passes.  When every cell equal to the
// threshold is selected the last pass only compares; otherwise the equal cells are ranked by
// index (per-chunk counts, their scan, and warp ballots within each chunk), as in many 256^3
// fields, where FP32 values near the threshold repeat (halo proxy and bias fit 305 us without the
// ranking and 330 with it).
//
// Bound by the reads of the field: at 256^3 three histogram passes and one comparing pass.  With
// eight-bit digits chosen on the host (four passes, four synchronisations) and a ranking pass
// always, the selection took 250 us there.
#include <algorithm>

#include "internal.h"
#include "particles.h"

namespace pm {

template <typename T> struct KeyOf;
template <> struct KeyOf<float> {
    typedef uint32_t K;
    static constexpr int BITS = 32;
    __device__ __forceinline__ static K key(float f) {
        const uint32_t u = __float_as_uint(f);
        return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    }
};
template <> struct KeyOf<double> {
    typedef unsigned long long K;
    static constexpr int BITS = 64;
    __device__ __forceinline__ static K key(double f) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(f);
        return (u & 0x8000000000000000ull) ? ~u : (u | 0x8000000000000000ull);
    }
};

constexpr int kDigitBits = 11, kDigits = 1 << kDigitBits;

// The state of a selection on the device.
struct SelectState {
    unsigned long long prefix, pmask;  // digits chosen so far and their mask
    unsigned long long remaining;      // places left among the cells that match the prefix
    unsigned long long equal;          // cells equal to the whole key (after the last digit)
};

// Four values a load where the field's address allows (`f` on a 16- or 32-byte boundary).
template <typename T> struct alignas(4 * sizeof(T)) Quad { T v[4]; };

// f(i, value) for every cell, in vectors of four when quads is set.
template <typename T, class F>
__device__ __forceinline__ void for_cells(const T* __restrict__ f, int64_t count, bool quads, F fn) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if (quads) {
        const int64_t n4 = count / 4;
        for (int64_t i = t0; i < n4; i += step) {
            const Quad<T> q = reinterpret_cast<const Quad<T>*>(f)[i];
#pragma unroll
            for (int w = 0; w < 4; ++w) fn(4 * i + w, q.v[w]);
        }
        done = 4 * n4;
    }
    for (int64_t i = done + t0; i < count; i += step) fn(i, f[i]);
}

template <typename T>
__global__ void __launch_bounds__(512) k_radix_hist(const T* __restrict__ f, int64_t count, bool quads,
                                                    const SelectState* __restrict__ st, int shift, int bits,
                                                    uint32_t* __restrict__ hist) {
    __shared__ uint32_t h[kDigits];
    for (int i = threadIdx.x; i < kDigits; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const unsigned long long prefix = st->prefix, pmask = st->pmask, dmask = (1ull << bits) - 1;
    for_cells(f, count, quads, [&](int64_t, T v) {
        const unsigned long long k = (unsigned long long)KeyOf<T>::key(v);
        if ((k & pmask) == prefix) atomicAdd(&h[(k >> shift) & dmask], 1u);
    });
    __syncthreads();
    for (int i = threadIdx.x; i < kDigits; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

// Chooses the digit whose cells, from the top, reach the remaining places, and clears the
// histogram for the next pass (one CTA; thread t holds the two digits 2 t, 2 t + 1).
__global__ void __launch_bounds__(1024) k_pick_digit(SelectState* __restrict__ st, int shift, int bits,
                                                     uint32_t* __restrict__ hist) {
    __shared__ unsigned long long warp_tot[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned long long remaining = st->remaining;
    // from the top: thread 0 takes the two largest digits
    const int hi = kDigits - 1 - 2 * t, lo = hi - 1;
    const unsigned long long ch = hist[hi], cl = hist[lo];
    hist[hi] = 0;
    hist[lo] = 0;
    unsigned long long incl = ch + cl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    unsigned long long before = incl - (ch + cl);
    for (int v = 0; v < w; ++v) before += warp_tot[v];
    int digit = -1;
    unsigned long long above = 0, equal = 0;
    if (before < remaining && before + ch >= remaining) digit = hi, above = before, equal = ch;
    else if (before + ch < remaining && before + ch + cl >= remaining) digit = lo, above = before + ch, equal = cl;
    if (digit >= 0) {  // one thread
        st->prefix |= (unsigned long long)digit << shift;
        st->pmask |= ((1ull << bits) - 1) << shift;
        st->remaining = remaining - above;
        st->equal = equal;
    }
}

// Cells equal to the threshold key are ranked by index without a full-length scan: CTA b
// owns the contiguous chunk [b chunk, (b + 1) chunk); k_eq_count counts its equal cells,
// a small scan over the CTAs gives each chunk its first rank, and k_select walks its chunk
// in index order, ranking the equal cells of each 256-cell tile with warp ballots.  None of the
// three does anything when all equal cells are selected.
template <typename T>
__global__ void __launch_bounds__(256) k_eq_count(const T* __restrict__ f, int64_t count, int64_t chunk,
                                                   const SelectState* __restrict__ st, uint32_t* __restrict__ cnt) {
    if (st->equal == st->remaining) return;
    const unsigned long long thr = st->prefix;
    __shared__ uint32_t wsum[8];
    const int64_t lo = (int64_t)blockIdx.x * chunk, hi = min(count, lo + chunk);
    uint32_t c = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x)
        c += ((unsigned long long)KeyOf<T>::key(f[i]) == thr) ? 1u : 0u;
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += wsum[w];
        cnt[blockIdx.x] = s;
    }
}

// In place: cnt[b] <- sum of cnt[0..b) (one CTA; nb is a few thousand).
__global__ void __launch_bounds__(1024) k_scan_small(uint32_t* __restrict__ cnt, int nb,
                                                     const SelectState* __restrict__ st) {
    if (st->equal == st->remaining) return;
    __shared__ uint32_t part[1024];
    const int per = (nb + 1023) / 1024, lo = threadIdx.x * per, hi = min(nb, lo + per);
    uint32_t s = 0;
    for (int i = lo; i < hi; ++i) s += cnt[i];
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int t = 0; t < 1024; ++t) {
            const uint32_t v = part[t];
            part[t] = run;
            run += v;
        }
    }
    __syncthreads();
    uint32_t run = part[threadIdx.x];
    for (int i = lo; i < hi; ++i) {
        const uint32_t v = cnt[i];
        cnt[i] = run;
        run += v;
    }
}

// delta_h = 1[selected] n^3/K - 1
template <typename T>
__global__ void __launch_bounds__(256) k_select(const T* __restrict__ f, int64_t count, int64_t chunk, bool quads,
                                                 const SelectState* __restrict__ st, const uint32_t* __restrict__ first,
                                                 T scale, T* __restrict__ out) {
    const unsigned long long thr = st->prefix, eq_needed = st->remaining;
    if (st->equal == eq_needed) {
        const T yes = scale - T(1);
        if (quads) {
            const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
            for (int64_t i = t0; i < count / 4; i += step) {
                const Quad<T> q = reinterpret_cast<const Quad<T>*>(f)[i];
                Quad<T> o;
#pragma unroll
                for (int w = 0; w < 4; ++w) o.v[w] = (unsigned long long)KeyOf<T>::key(q.v[w]) >= thr ? yes : T(-1);
                reinterpret_cast<Quad<T>*>(out)[i] = o;
            }
        }
        for_cells(f + (quads ? count / 4 * 4 : 0), quads ? count % 4 : count, false, [&](int64_t i, T v) {
            out[(quads ? count / 4 * 4 : 0) + i] = (unsigned long long)KeyOf<T>::key(v) >= thr ? yes : T(-1);
        });
        return;
    }
    __shared__ uint32_t wcnt[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int64_t lo = (int64_t)blockIdx.x * chunk, hi = min(count, lo + chunk);
    uint32_t base = first[blockIdx.x];  // rank of the chunk's first equal cell
    for (int64_t t0 = lo; t0 < hi; t0 += blockDim.x) {
        const int64_t i = t0 + threadIdx.x;
        unsigned long long k = 0;
        bool eq = false;
        if (i < hi) {
            k = (unsigned long long)KeyOf<T>::key(f[i]);
            eq = k == thr;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, eq);
        if (lane == 0) wcnt[w] = __popc(bal);
        __syncthreads();
        uint32_t before = base;
        for (int v = 0; v < w; ++v) before += wcnt[v];
        uint32_t tile = 0;
        for (int v = 0; v < nw; ++v) tile += wcnt[v];
        if (i < hi) {
            const uint32_t rank = before + __popc(bal & ((1u << lane) - 1u));
            const bool sel = k > thr || (eq && rank < eq_needed);
            out[i] = sel ? scale - T(1) : T(-1);
        }
        base += tile;
        __syncthreads();  // wcnt is rewritten by the next tile
    }
}

__global__ void k_select_start(SelectState* __restrict__ st, unsigned long long K, uint32_t* __restrict__ hist) {
    for (int i = threadIdx.x; i < kDigits; i += blockDim.x) hist[i] = 0;
    if (threadIdx.x == 0) *st = SelectState{0, 0, K, 0};
}

static unsigned blocks_for(int64_t count) {
    int64_t b = (count + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    return (unsigned)(b < 1 ? 1 : b);
}

template <typename T>
cudaError_t halo_proxy(const T* field, int64_t count, int64_t K, T* out, void* scratch, cudaStream_t st) {
    SelectState* state = (SelectState*)scratch;
    uint32_t* hist = (uint32_t*)((char*)scratch + 256);
    uint32_t* first = hist + kDigits;  // per-CTA counts
    const uintptr_t align = 4 * sizeof(T) - 1;
    const bool in4 = ((uintptr_t)field & align) == 0, both4 = in4 && ((uintptr_t)out & align) == 0;
    const unsigned nb = blocks_for(count);
    const int64_t chunk = (count + nb - 1) / nb;
    // 512 threads with four cells each
    const unsigned nh = (unsigned)std::min<int64_t>((count + 2047) / 2048, 152 * 4);
    k_select_start<<<1, 256, 0, st>>>(state, (unsigned long long)K, hist);
    for (int top = KeyOf<T>::BITS; top > 0;) {
        const int bits = top < kDigitBits ? top : kDigitBits, shift = top - bits;
        k_radix_hist<T><<<nh, 512, 0, st>>>(field, count, in4, state, shift, bits, hist);
        k_pick_digit<<<1, 1024, 0, st>>>(state, shift, bits, hist);
        top = shift;
    }
    k_eq_count<T><<<nb, 256, 0, st>>>(field, count, chunk, state, first);
    k_scan_small<<<1, 1024, 0, st>>>(first, (int)nb, state);
    k_select<T><<<nb, 256, 0, st>>>(field, count, chunk, both4, state, first, (T)((double)count / (double)K), out);
    return cudaGetLastError();
}

size_t halo_proxy_scratch_bytes(int64_t count) {
    return 256 + sizeof(uint32_t) * ((size_t)kDigits + blocks_for(count));
}

template cudaError_t halo_proxy<float>(const float*, int64_t, int64_t, float*, void*, cudaStream_t);
template cudaError_t halo_proxy<double>(const double*, int64_t, int64_t, double*, void*, cudaStream_t);

}  // namespace pm

// Particle-side kernels of the PM step: CIC deposit (counting density, Sec. 4), CIC
// interpolation and the unfused kick + drift (KDK in a; the fused update with the next
// deposit is in update.cu), Zel'dovich placement, the per-wavevector Philox phases, the GR
// displacement combination (Eqs. xiGR and combined) and the cell keys / stable cell order
// of the particles.
//
// Position encodings (units of the box side):
//   FP32 path: uint32 ticks, 2^32 per side; the periodic wrap is integer overflow.
//   FP64 path: double fraction in [0, 1).
// Mesh nodes sit at cell centres, so mesh coordinate s = x n - 1/2; on ticks that
// is (u - 2^(31 - log2 n)) >> (32 - log2 n) for the base node and the low bits
// for the fraction, both exact.
#include <math.h>

#include <mutex>
#include <type_traits>

#include "dfloat.cuh"
#include "internal.h"
#include "particles.h"
#include "update_dev.cuh"

namespace pm {

// ---------------------------------------------------------------- CIC decode (FP64 fractions)
// Base node, its neighbour and the two weights along one axis of s = x n - 1/2 (n = 2^logn).
// FP64 arithmetic bounds the FP64 particle kernels (its pipe is 84-87% busy), so for x n >= 1 the
// decode is done on the bits: x n is its mantissa shifted into units of 2^-52, where subtracting
// 1/2 and splitting off the fraction are exact, as they are in FP64, and two FP64 subtractions
// give the weights.  In the first cell, which most warps meet on small meshes, the base is known
// from the sign of s and three operations give the weights; positions outside [0, 1) take the
// general form.
struct CicD {
    int i0, i1;
    double w0, w1;
};
// (Out of line, so that its FP64 instructions are not issued for the others' predicates.)
__device__ __noinline__ CicD cic_frac_general(double x, int logn) {
    CicD c;
    const int n = 1 << logn;
    const double s = x * __hiloint2double((1023 + logn) << 20, 0) - 0.5;  // x n - 1/2
    if ((unsigned)__double2hiint(x) < (unsigned)(1023 - logn) << 20) {    // 0 <= x n < 1
        const bool below = __double2hiint(s) < 0;
        c.w1 = below ? s + 1.0 : s;
        c.i0 = below ? n - 1 : 0;
    } else {
        const double fl = floor(s);
        c.w1 = s - fl;
        c.i0 = ((int)fl) & (n - 1);
    }
    c.w0 = 1.0 - c.w1;
    c.i1 = (c.i0 + 1) & (n - 1);
    return c;
}
__device__ __forceinline__ CicD cic_frac(double x, int logn) {
    const int n = 1 << logn;
    CicD c;
    const long long bits = __double_as_longlong(x);
    const int e = (int)(bits >> 52) - 1023 + logn;  // exponent of x n (the sign makes it large)
    if ((unsigned)e < (unsigned)logn) {
        const long long m = bits & 0xfffffffffffffll;
        const long long v = ((m | (1ll << 52)) << e) - (1ll << 51);
        c.i0 = (int)(v >> 52);
        const double d = __longlong_as_double((v & 0xfffffffffffffll) | 0x3ff0000000000000ll);  // 1 + fraction
        c.w1 = d - 1.0;
        c.w0 = 2.0 - d;
        c.i1 = (c.i0 + 1) & (n - 1);
    } else {
        c = cic_frac_general(x, logn);
    }
    return c;
}

// ---------------------------------------------------------------- deposit
// The vector forms below read and write aligned groups of four cells of a z row: rows of at least
// one such group, on 16-byte boundaries.
static bool quad_rows(const void* mesh, int n) { return n >= 4 && (uintptr_t)mesh % 16 == 0; }

// Particles in any order.  Bound by the L2's atomic operations: with V4 (quad_rows) the
// two z corners of a row go in one vector reduction when they share an aligned group of four
// cells (three rows in four), its other lanes adding 0.
template <bool V4>
__global__ void __launch_bounds__(256) k_deposit_ticks(const uint32_t* __restrict__ x, int64_t count, int logn,
                                                       float inv_cell_ticks, float mass, float* __restrict__ rho) {
    const size_t n = (size_t)1 << logn;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const CicF cx = cic_ticks(x[i], logn, inv_cell_ticks);
        const CicF cy = cic_ticks(x[count + i], logn, inv_cell_ticks);
        const CicF cz = cic_ticks(x[2 * count + i], logn, inv_cell_ticks);
        const float wx[2] = {1.0f - cx.w1, cx.w1}, wy[2] = {1.0f - cy.w1, cy.w1}, wz[2] = {1.0f - cz.w1, cz.w1};
        const int ix[2] = {cx.i0, cx.i1}, iy[2] = {cy.i0, cy.i1}, iz[2] = {cz.i0, cz.i1};
        const int pos = cz.i0 & 3;
        if (V4 && pos != 3) {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float wab = mass * wx[a] * wy[b], v0 = wab * wz[0], v1 = wab * wz[1];
                    red_add_v4(rho + ((size_t)ix[a] * n + iy[b]) * n + (cz.i0 - pos),
                               make_float4(pos == 0 ? v0 : 0.f, pos == 0 ? v1 : pos == 1 ? v0 : 0.f,
                                           pos == 1 ? v1 : pos == 2 ? v0 : 0.f, pos == 2 ? v1 : 0.f));
                }
        } else {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const float wab = mass * wx[a] * wy[b];
                    float* row = rho + ((size_t)ix[a] * n + iy[b]) * n;
                    atomicAdd(row + iz[0], wab * wz[0]);
                    atomicAdd(row + iz[1], wab * wz[1]);
                }
        }
    }
}

// blockIdx.y selects the field of a batch (particles [field][3][np^3], meshes [field][n^3]).
template <int R, int XC>
__global__ void __launch_bounds__(512, 3) k_deposit_tiled(const uint32_t* __restrict__ x, int lognp, int logn,
                                                          float inv_cell_ticks, float mass, float* __restrict__ rho) {
    typedef DepTile<R, XC> D;
    extern __shared__ __align__(16) uint32_t lo[];  // D::CELLS
    x += (int64_t)blockIdx.y * 3 << (3 * lognp);
    rho += (int64_t)blockIdx.y << (3 * logn);
    const int ntz = (1 << lognp) / D::TZ, nty = (1 << lognp) / D::TY;
    const int bz = blockIdx.x % ntz, by = (blockIdx.x / ntz) % nty, bx = blockIdx.x / (ntz * nty);
    const int ox = D::box_x(bx), oy = by * D::TY * R - D::H, oz = bz * D::TZ * R - D::HZ;
    const int64_t count = (int64_t)1 << (3 * lognp);
    tile_zero<D::CELLS>(lo);
    __syncthreads();
    auto pid = [&](int e) -> int64_t {
        const int lz = e % D::TZ, ly = (e / D::TZ) % D::TY, lx = e / (D::TZ * D::TY);
        return ((((int64_t)(bx * D::TX + lx) << lognp) + by * D::TY + ly) << lognp) + bz * D::TZ + lz;
    };
    const float quanta = mass * kTileQuanta;
    TileAdds adds;
    // positions are loaded one iteration ahead (their latency overlaps the deposit)
    int64_t idn = pid(threadIdx.x);
    uint32_t nu0 = 0, nu1 = 0, nu2 = 0;
    if (D::PER >= 512 || threadIdx.x < D::PER) nu0 = x[idn], nu1 = x[count + idn], nu2 = x[2 * count + idn];
#pragma unroll 1
    for (int e = threadIdx.x; e < D::PER; e += 512) {
        const uint32_t u0 = nu0, u1 = nu1, u2 = nu2;
        if (e + 512 < D::PER) {
            idn = pid(e + 512);
            nu0 = x[idn];
            nu1 = x[count + idn];
            nu2 = x[2 * count + idn];
        }
        tile_deposit<D, false>(lo, rho, u0, u1, u2, logn, inv_cell_ticks, ox, oy, oz, quanta, adds);
    }
    tile_close<D>(lo, rho, ox, oy, oz, logn, adds, [&] {
        tile_again<D>(lo, rho, ox, oy, oz, logn, [&] {
            for (int e = threadIdx.x; e < D::PER; e += 512) {
                const int64_t id = pid(e);
                tile_deposit<D, true>(lo, rho, x[id], x[count + id], x[2 * count + id], logn, inv_cell_ticks, ox, oy,
                                      oz, quanta, adds);
            }
        });
    });
}

// R = 1: each thread walks one lattice row of the CTA's block along x and carries the upper-x
// plane of its CIC stencil to the next particle (the deposit half of the fused update kernel).
template <int XC>
__global__ void __launch_bounds__(512, 3) k_deposit_sweep(const uint32_t* __restrict__ x, int lognp, int logn,
                                                          float inv_cell_ticks, float mass, float* __restrict__ rho) {
    typedef DepTile<1, XC> D;
    static_assert(D::TY * D::TZ == 512, "one thread per (ly, lz); lx runs over the loop");
    extern __shared__ __align__(16) uint32_t lo[];  // D::CELLS
    x += (int64_t)blockIdx.y * 3 << (3 * lognp);
    rho += (int64_t)blockIdx.y << (3 * logn);
    const int np = 1 << lognp;
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int ntz = np / D::TZ, nty = np / D::TY;
    const int bz = blockIdx.x % ntz, by = (blockIdx.x / ntz) % nty, bx = blockIdx.x / (ntz * nty);
    const int ox = D::box_x(bx), oy = by * D::TY - D::H, oz = bz * D::TZ - D::HZ;
    tile_zero<D::CELLS>(lo);
    __syncthreads();
    const int lz = threadIdx.x % D::TZ, ly = threadIdx.x / D::TZ;
    const int64_t id0 = ((((int64_t)(bx * D::TX) << lognp) + by * D::TY + ly) << lognp) + bz * D::TZ + lz;
    const int64_t xstride = (int64_t)1 << (2 * lognp);
    const float quanta = mass * kTileQuanta;
    SweepCarry sc;
    uint32_t nu0 = x[id0], nu1 = x[count + id0], nu2 = x[2 * count + id0];
#pragma unroll 1
    for (int lx = 0; lx < D::TX; ++lx) {
        const uint32_t u0 = nu0, u1 = nu1, u2 = nu2;
        if (lx + 1 < D::TX) {
            const int64_t idn = id0 + (lx + 1) * xstride;
            nu0 = x[idn];
            nu1 = x[count + idn];
            nu2 = x[2 * count + idn];
        }
        sweep_deposit<D>(lo, rho, u0, u1, u2, logn, inv_cell_ticks, ox, oy, oz, quanta, sc);
    }
    if (sc.dnext >= 0) sweep_carried<D>(lo, sc);
    tile_close<D>(lo, rho, ox, oy, oz, logn, sc.adds, [&] {
        tile_again<D>(lo, rho, ox, oy, oz, logn, [&] {
            for (int lx = 0; lx < D::TX; ++lx) {
                const int64_t id = id0 + lx * xstride;
                tile_deposit<D, true>(lo, rho, x[id], x[count + id], x[2 * count + id], logn, inv_cell_ticks, ox, oy,
                                      oz, quanta, sc.adds);
            }
        });
    });
}

__global__ void k_deposit_frac(const double* __restrict__ x, int64_t count, int logn, double mass,
                               double* __restrict__ rho) {
    const size_t n = (size_t)1 << logn;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        CicD cx = cic_frac(x[i], logn);
        const CicD cy = cic_frac(x[count + i], logn), cz = cic_frac(x[2 * count + i], logn);
        if (mass != 1.0) cx.w0 *= mass, cx.w1 *= mass;
        const double wx[2] = {cx.w0, cx.w1}, wy[2] = {cy.w0, cy.w1};
        const int ix[2] = {cx.i0, cx.i1}, iy[2] = {cy.i0, cy.i1};
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const double wab = wx[a] * wy[b];
                double* row = rho + ((size_t)ix[a] * n + iy[b]) * n;
                atomicAdd(row + cz.i0, wab * cz.w0);
                atomicAdd(row + cz.i1, wab * cz.w1);
            }
    }
}

// The np^3 = n^3 lattice-ordered particles of a context: a thread walks a lattice row along x in
// runs of `run` and carries the upper plane's weights to the next particle, which usually starts
// one cell further: 4 atomics a particle instead of 8 (the FP64 atomics bound the plain form).
__global__ void __launch_bounds__(256) k_deposit_frac_rows(const double* __restrict__ x, int logn, int run,
                                                           double* __restrict__ rho) {
    const int n = 1 << logn;
    const int64_t count = (int64_t)1 << (3 * logn), xstride = (int64_t)1 << (2 * logn);
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lx0 = (int)(gid >> (2 * logn)) * run;
    if (lx0 >= n) return;
    int64_t i = ((int64_t)lx0 << (2 * logn)) + (gid & (xstride - 1));
    uint32_t next = 0xffffffffu, o[4] = {0u, 0u, 0u, 0u};  // the carried plane's cell and corners
    double W[4];
#pragma unroll 1
    for (int k = 0; k < run; ++k, i += xstride) {
        const CicD cx = cic_frac(x[i], logn), cy = cic_frac(x[count + i], logn), cz = cic_frac(x[2 * count + i], logn);
        const uint32_t yz = ((uint32_t)cy.i0 << logn) | (uint32_t)cz.i0;
        const bool merge = (((uint32_t)cx.i0 << (2 * logn)) | yz) == next;
        if (!merge && next != 0xffffffffu) {
#pragma unroll
            for (int q = 0; q < 4; ++q) atomicAdd(rho + o[q], W[q]);
        }
        next = ((uint32_t)cx.i1 << (2 * logn)) | yz;
        const double wy[2] = {cy.w0, cy.w1}, wz[2] = {cz.w0, cz.w1};
        const uint32_t iy[2] = {(uint32_t)cy.i0, (uint32_t)cy.i1}, iz[2] = {(uint32_t)cz.i0, (uint32_t)cz.i1};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double w = wy[q >> 1] * wz[q & 1];
            const double lower = merge ? fma(cx.w0, w, W[q]) : cx.w0 * w;
            atomicAdd(rho + ((((uint32_t)cx.i0 << logn) + iy[q >> 1]) << logn) + iz[q & 1], lower);
            W[q] = cx.w1 * w;
            o[q] = ((((uint32_t)cx.i1 << logn) + iy[q >> 1]) << logn) + iz[q & 1];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) atomicAdd(rho + o[q], W[q]);
}

static unsigned grid_for(int64_t count, int threads) {
    int64_t b = (count + threads - 1) / threads;
    const int64_t cap = 152 * 32;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

template <int R, int XC>
static cudaError_t deposit_tiled_r(const void* x, int np, int n, double mass, void* rho, cudaStream_t st, int nfields) {
    typedef DepTile<R, XC> D;
    const int lognp = ilog2(np), logn = ilog2(n);
    const unsigned blocks = (unsigned)((np / D::TX) * (np / D::TY) * (np / D::TZ));
    const float inv = (float)ldexp(1.0, -(32 - logn));
    const size_t smem = sizeof(uint32_t) * D::CELLS;
    const auto fn = [] {
        if constexpr (R == 1) return k_deposit_sweep<XC>;
        else return k_deposit_tiled<R, XC>;
    }();
    cudaError_t e = set_smem_once((const void*)fn, smem);
    if (e != cudaSuccess) return e;
    fn<<<dim3(blocks, nfields), 512, smem, st>>>((const uint32_t*)x, lognp, logn, inv, (float)mass, (float*)rho);
    return cudaGetLastError();
}
template <int R>
static cudaError_t deposit_tiled(const void* x, int np, int n, double mass, void* rho, cudaStream_t st, int nfields) {
    switch (tile_depth(R, np, nfields)) {
        case 2: return deposit_tiled_r<R, R == 4 ? 4 : 2>(x, np, n, mass, rho, st, nfields);
        case 4: return deposit_tiled_r<R, 4>(x, np, n, mass, rho, st, nfields);
        case 8: return deposit_tiled_r<R, 8>(x, np, n, mass, rho, st, nfields);
        default: return deposit_tiled_r<R, 16>(x, np, n, mass, rho, st, nfields);
    }
}

cudaError_t deposit_lattice(const void* x, int np, int precision, int n, double mass, void* rho, cudaStream_t st,
                            int nfields) {
    const int R = n / np;
    // the tile box (16 + 4) x (16 + 4) x (32 + 8) cells must fit in the mesh without overlapping itself
    const bool tiled = precision == PM_FP32_FIXED && n >= 64 && (R == 1 || R == 2 || R == 4) && np >= 32 / R &&
                       (uintptr_t)rho % 16 == 0;
    if (!tiled) {
        if (nfields != 1) return cudaErrorInvalidValue;
        if (precision == PM_FP64 && R == 1 && mass == 1.0) {
            // rows of 16 while they still give every SM two blocks; on lattices too small for rows
            // of four (64^3: two) the particles by themselves are as fast or faster (64^3: 20.5 us
            // against 22.6)
            int run = 16;
            while (run > 1 && (int64_t)np * np * np / run < 2 * 256 * (int64_t)num_sms()) run /= 2;
            if (run < 4) return deposit(x, (int64_t)np * np * np, precision, n, mass, rho, st);
            k_deposit_frac_rows<<<(unsigned)((int64_t)np * np * (np / run) / 256), 256, 0, st>>>(
                (const double*)x, ilog2(n), run, (double*)rho);
            return cudaGetLastError();
        }
        return deposit(x, (int64_t)np * np * np, precision, n, mass, rho, st);
    }
    if (R == 1) return deposit_tiled<1>(x, np, n, mass, rho, st, nfields);
    if (R == 2) return deposit_tiled<2>(x, np, n, mass, rho, st, nfields);
    return deposit_tiled<4>(x, np, n, mass, rho, st, nfields);
}

cudaError_t deposit(const void* x, int64_t count, int precision, int n, double mass, void* rho,
                    cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    const int logn = ilog2(n);
    if (precision == PM_FP32_FIXED) {
        const float inv = (float)ldexp(1.0, -(32 - logn));
        const auto fn = quad_rows(rho, n) ? k_deposit_ticks<true> : k_deposit_ticks<false>;
        fn<<<grid_for(count, 256), 256, 0, st>>>((const uint32_t*)x, count, logn, inv, (float)mass, (float*)rho);
    } else {
        k_deposit_frac<<<grid_for(count, 256), 256, 0, st>>>((const double*)x, count, logn, mass, (double*)rho);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- interpolation
template <typename T>
__device__ __forceinline__ T gather8(const T* __restrict__ f, size_t n, const int* ix, const int* iy,
                                     const int* iz, const T* wx, const T* wy, const T* wz) {
    T acc = T(0);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const T* row = f + ((size_t)ix[a] * n + iy[b]) * n;
            acc += wx[a] * wy[b] * (wz[0] * __ldg(row + iz[0]) + wz[1] * __ldg(row + iz[1]));
        }
    return acc;
}

// V4 (quad_rows): a row's two z corners come in one 16-byte load when they share an
// aligned group of four cells, which saves requests to L2.
template <bool V4>
__global__ void k_interp_ticks(const float* __restrict__ f, int logn, const uint32_t* __restrict__ x,
                               int64_t count, float inv_cell_ticks, float* __restrict__ out) {
    const size_t n = (size_t)1 << logn;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const CicF cx = cic_ticks(x[i], logn, inv_cell_ticks);
        const CicF cy = cic_ticks(x[count + i], logn, inv_cell_ticks);
        const CicF cz = cic_ticks(x[2 * count + i], logn, inv_cell_ticks);
        const float wx[2] = {1.0f - cx.w1, cx.w1}, wy[2] = {1.0f - cy.w1, cy.w1}, wz[2] = {1.0f - cz.w1, cz.w1};
        const int ix[2] = {cx.i0, cx.i1}, iy[2] = {cy.i0, cy.i1}, iz[2] = {cz.i0, cz.i1};
        if constexpr (V4) {
            const int pos = cz.i0 & 3;
            float4 v[4];
            float next[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float* row = f + ((size_t)ix[q >> 1] * n + iy[q & 1]) * n;
                v[q] = __ldg(reinterpret_cast<const float4*>(row + (cz.i0 - pos)));
                next[q] = pos == 3 ? __ldg(row + cz.i1) : 0.f;
            }
            float acc = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float f0 = pos == 0 ? v[q].x : pos == 1 ? v[q].y : pos == 2 ? v[q].z : v[q].w;
                const float f1 = pos == 0 ? v[q].y : pos == 1 ? v[q].z : pos == 2 ? v[q].w : next[q];
                acc += wx[q >> 1] * wy[q & 1] * (wz[0] * f0 + wz[1] * f1);
            }
            out[i] = acc;
        } else {
            out[i] = gather8<float>(f, n, ix, iy, iz, wx, wy, wz);
        }
    }
}

__global__ void k_interp_frac(const double* __restrict__ f, int logn, const double* __restrict__ x, int64_t count,
                              double* __restrict__ out) {
    const size_t n = (size_t)1 << logn;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const CicD cx = cic_frac(x[i], logn), cy = cic_frac(x[count + i], logn), cz = cic_frac(x[2 * count + i], logn);
        const double wx[2] = {cx.w0, cx.w1}, wy[2] = {cy.w0, cy.w1}, wz[2] = {cz.w0, cz.w1};
        const int ix[2] = {cx.i0, cx.i1}, iy[2] = {cy.i0, cy.i1}, iz[2] = {cz.i0, cz.i1};
        out[i] = gather8<double>(f, n, ix, iy, iz, wx, wy, wz);
    }
}

cudaError_t interp(const void* field, int n, const void* x, int64_t count, int precision, void* out,
                   cudaStream_t st) {
    if (count == 0) return cudaSuccess;
    const int logn = ilog2(n);
    if (precision == PM_FP32_FIXED) {
        const float inv = (float)ldexp(1.0, -(32 - logn));
        const auto fn = quad_rows(field, n) ? k_interp_ticks<true> : k_interp_ticks<false>;
        fn<<<grid_for(count, 256), 256, 0, st>>>((const float*)field, logn, (const uint32_t*)x, count, inv, (float*)out);
    } else {
        k_interp_frac<<<grid_for(count, 256), 256, 0, st>>>((const double*)field, logn, (const double*)x, count,
                                                            (double*)out);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- interp + kick + drift
template <bool FD>
__global__ void __launch_bounds__(256) k_ikd_ticks(uint32_t* __restrict__ x, float* __restrict__ p, int64_t count,
                                                   int logn, float inv_cell_ticks, const float* __restrict__ g,
                                                   float kick, float drift_ticks, float inv_d) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t u0 = x[i], u1 = x[count + i], u2 = x[2 * count + i];
        float p0 = p[i], p1 = p[count + i], p2 = p[2 * count + i];
        ikd_particle<FD>(u0, u1, u2, p0, p1, p2, logn, inv_cell_ticks, g, kick, drift_ticks, inv_d);
        p[i] = p0;
        p[count + i] = p1;
        p[2 * count + i] = p2;
        x[i] = u0;
        x[count + i] = u1;
        x[2 * count + i] = u2;
    }
}

// Same update, two neighbouring particles per thread through 8-byte loads and stores
// (count even, arrays 8-byte aligned): neighbours share most CIC corners, so the
// second particle's gathers mostly hit L1.
template <bool FD>
__global__ void __launch_bounds__(256) k_ikd_ticks2(uint32_t* __restrict__ x, float* __restrict__ p, int64_t count,
                                                    int logn, float inv_cell_ticks, const float* __restrict__ g,
                                                    float kick, float drift_ticks, float inv_d) {
    const int64_t pairs = count >> 1;
    uint2* x0 = reinterpret_cast<uint2*>(x);
    uint2* x1 = reinterpret_cast<uint2*>(x + count);
    uint2* x2 = reinterpret_cast<uint2*>(x + 2 * count);
    float2* p0 = reinterpret_cast<float2*>(p);
    float2* p1 = reinterpret_cast<float2*>(p + count);
    float2* p2 = reinterpret_cast<float2*>(p + 2 * count);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pairs;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint2 a = x0[i], b = x1[i], c = x2[i];
        float2 pa = p0[i], pb = p1[i], pc = p2[i];
        ikd_particle<FD>(a.x, b.x, c.x, pa.x, pb.x, pc.x, logn, inv_cell_ticks, g, kick, drift_ticks, inv_d);
        ikd_particle<FD>(a.y, b.y, c.y, pa.y, pb.y, pc.y, logn, inv_cell_ticks, g, kick, drift_ticks, inv_d);
        p0[i] = pa;
        p1[i] = pb;
        p2[i] = pc;
        x0[i] = a;
        x1[i] = b;
        x2[i] = c;
    }
}

// A box fraction wrapped into [0, 1): the integer part is only taken off when there is one (out
// of line, as above).
__device__ __noinline__ double minus_floor(double x) { return x - floor(x); }
__device__ __forceinline__ double wrap_fraction(double x) {
    if ((unsigned)__double2hiint(x) >= 0x3ff00000u) x = minus_floor(x);
    return x;
}

template <bool FD>
__global__ void __launch_bounds__(256) k_ikd_frac(double* __restrict__ x, double* __restrict__ p, int64_t count,
                                                  int logn, const double* __restrict__ g, double kick, double drift_box,
                                                  double inv_d) {
    const size_t n = (size_t)1 << logn;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        double xs[3] = {x[i], x[count + i], x[2 * count + i]};
        const CicD cx = cic_frac(xs[0], logn), cy = cic_frac(xs[1], logn), cz = cic_frac(xs[2], logn);
        const double wx[2] = {cx.w0, cx.w1}, wy[2] = {cy.w0, cy.w1}, wz[2] = {cz.w0, cz.w1};
        const int ix[2] = {cx.i0, cx.i1}, iy[2] = {cy.i0, cy.i1}, iz[2] = {cz.i0, cz.i1};
        double f[3] = {0.0, 0.0, 0.0};
        if constexpr (FD) {
            double P[2][4];
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b)
#pragma unroll
                    for (int c = 0; c < 2; ++c) P[a][2 * b + c] = g[((size_t)ix[a] * n + iy[b]) * n + iz[c]];
            fd1_force<double>(P[0], P[1], wx[0], wx[1], wy, wz, inv_d, f[0], f[1], f[2]);
        } else {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const double wab = wx[a] * wy[b];
                    const double* row = g + ((size_t)ix[a] * n + iy[b]) * n * kForceRows;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const double w = wab * wz[c];
#pragma unroll
                        for (int j = 0; j < 3; ++j) f[j] = fma(w, __ldg(row + j * n + iz[c]), f[j]);
                    }
                }
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double pj = p[j * count + i] + kick * f[j];
            p[j * count + i] = pj;
            x[j * count + i] = wrap_fraction(xs[j] + drift_box * pj);
        }
    }
}

template <bool FD>
static cudaError_t interp_kick_drift_t(void* x, void* p, int64_t count, int precision, int n, const void* g,
                                       double kick, double drift, double box, double inv_d, cudaStream_t st) {
    const int logn = ilog2(n);
    if (precision == PM_FP32_FIXED) {
        const float inv = (float)ldexp(1.0, -(32 - logn));
        const float dt = (float)(drift * (4294967296.0 / box));
        const bool pairs = (count % 2 == 0) && ((uintptr_t)x % 8 == 0) && ((uintptr_t)p % 8 == 0);
        if (pairs)
            k_ikd_ticks2<FD><<<grid_for(count / 2, 256), 256, 0, st>>>((uint32_t*)x, (float*)p, count, logn, inv,
                                                                       (const float*)g, (float)kick, dt,
                                                                       (float)inv_d);
        else
            k_ikd_ticks<FD><<<grid_for(count, 256), 256, 0, st>>>((uint32_t*)x, (float*)p, count, logn, inv,
                                                                  (const float*)g, (float)kick, dt, (float)inv_d);
    } else {
        k_ikd_frac<FD><<<grid_for(count, 256), 256, 0, st>>>((double*)x, (double*)p, count, logn, (const double*)g, kick,
                                                             drift / box, inv_d);
    }
    return cudaGetLastError();
}

cudaError_t interp_kick_drift(void* x, void* p, int64_t count, int precision, int n, const void* g,
                              double kick, double drift, double box, cudaStream_t st, double fd_inv_d) {
    if (count == 0) return cudaSuccess;
    if (fd_inv_d > 0.0) return interp_kick_drift_t<true>(x, p, count, precision, n, g, kick, drift, box, fd_inv_d, st);
    return interp_kick_drift_t<false>(x, p, count, precision, n, g, kick, drift, box, 0.0, st);
}

// ---------------------------------------------------------------- Zel'dovich placement
// x = q + D Psi(q), p = a^2 E f D Psi(q); q the lattice node of particle id i.  The FP32 path
// multiplies by pairs (dfloat.cuh) instead of in FP64: at 512^3 the FP64 products and their
// conversions took 3.6 ms for 4.8 GB moved.
// The displacement in ticks: the pair rounded to the nearest integer; beyond 2^30 ticks (a
// quarter of the box) in FP64, whose 64-bit conversion wraps like the positions.
struct TickScale {
    df f;
    double d;
};
__device__ __noinline__ uint32_t wrapped_ticks(float p1, double s1, float p2, double s2) {
    return (uint32_t)__double2ll_rn((double)p1 * s1 + (double)p2 * s2);
}
__device__ __forceinline__ uint32_t disp_ticks(float ps, const TickScale& s) {
    df v = two_prod(ps, s.f.h);
    if (!(fabsf(v.h) < 1073741824.0f)) return wrapped_ticks(ps, s.d, 0.0f, 0.0);
    v.l = fmaf(ps, s.f.l, v.l);
    return (uint32_t)df2int_rn(v);
}
// The two terms of the second-order placement.
__device__ __forceinline__ uint32_t disp_ticks(float p1, const TickScale& s1, float p2, const TickScale& s2) {
    df a = two_prod(p1, s1.f.h), b = two_prod(p2, s2.f.h);
    a.l = fmaf(p1, s1.f.l, a.l);
    b.l = fmaf(p2, s2.f.l, b.l);
    const df v = a + b;
    if (!(fabsf(a.h) < 1073741824.0f && fabsf(b.h) < 1073741824.0f && fabsf(v.h) < 1073741824.0f))
        return wrapped_ticks(p1, s1.d, p2, s2.d);
    return (uint32_t)df2int_rn(v);
}
static TickScale tick_scale(double d) { return TickScale{df_of(d), d}; }
// The scales of a launch's fields, made on the host as for a single run, so that a realisation's
// ticks are the single run's.
struct TickScales {
    static constexpr int MAX = 128;
    TickScale s[MAX];
};

// TickScales: blockIdx.y selects the field of a batch (particles [field][3][np^3], meshes
// [field][np^3]).  A single run's scale and arrays stay parameters: 28 registers instead of 40, and
// 0.12 ms of the 512^3 placement.
template <class Scales>
__global__ void k_ic_ticks(uint32_t* __restrict__ x, float* __restrict__ p, const float* __restrict__ psx,
                           const float* __restrict__ psy, const float* __restrict__ psz, int lognp,
                           const __grid_constant__ Scales scales, df pfac) {
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int sh = 32 - lognp;
    const int mask = (1 << lognp) - 1;
    TickScale scale;
    if constexpr (std::is_same<Scales, TickScales>::value) {
        scale = scales.s[blockIdx.y];
        x += blockIdx.y * 3 * count;
        p += blockIdx.y * 3 * count;
        psx += blockIdx.y * count;
        psy += blockIdx.y * count;
        psz += blockIdx.y * count;
    } else {
        scale = scales;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t q[3] = {(uint32_t)((i >> (2 * lognp)) & mask) << sh, (uint32_t)((i >> lognp) & mask) << sh,
                               (uint32_t)(i & mask) << sh};
        const float ps[3] = {psx[i], psy[i], psz[i]};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            x[j * count + i] = q[j] + disp_ticks(ps[j], scale);
            p[j * count + i] = fmaf(ps[j], pfac.h, ps[j] * pfac.l);
        }
    }
}

__global__ void k_ic_frac(double* __restrict__ x, double* __restrict__ p, const double* __restrict__ psx,
                          const double* __restrict__ psy, const double* __restrict__ psz, int lognp, double disp_box,
                          double pfac) {
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int mask = (1 << lognp) - 1;
    const double inv_np = ldexp(1.0, -lognp);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double q[3] = {(double)((i >> (2 * lognp)) & mask) * inv_np, (double)((i >> lognp) & mask) * inv_np,
                             (double)(i & mask) * inv_np};
        const double ps[3] = {psx[i], psy[i], psz[i]};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            double xj = q[j] + disp_box * ps[j];
            xj -= floor(xj);
            x[j * count + i] = xj;
            p[j * count + i] = pfac * ps[j];
        }
    }
}

cudaError_t ic_place(void* x, void* p, void* const* psi, int np, int precision, double D, double pfac, double box,
                     cudaStream_t st, int nfields, const double* boxes) {
    const int lognp = ilog2(np);
    const int64_t count = (int64_t)np * np * np;
    if (precision == PM_FP32_FIXED) {
        if (nfields == 1) {
            k_ic_ticks<<<grid_for(count, 256), 256, 0, st>>>((uint32_t*)x, (float*)p, (const float*)psi[0],
                                                             (const float*)psi[1], (const float*)psi[2], lognp,
                                                             tick_scale(D * 4294967296.0 / (boxes ? boxes[0] : box)),
                                                             df_of(pfac));
            return cudaGetLastError();
        }
        for (int f0 = 0; f0 < nfields; f0 += TickScales::MAX) {
            const int c = nfields - f0 < TickScales::MAX ? nfields - f0 : TickScales::MAX;
            TickScales s = {};
            for (int i = 0; i < c; ++i) s.s[i] = tick_scale(D * 4294967296.0 / boxes[f0 + i]);
            k_ic_ticks<<<dim3(grid_for(count, 256), c), 256, 0, st>>>(
                (uint32_t*)x + f0 * 3 * count, (float*)p + f0 * 3 * count, (const float*)psi[0] + f0 * count,
                (const float*)psi[1] + f0 * count, (const float*)psi[2] + f0 * count, lognp, s, df_of(pfac));
        }
    } else {
        k_ic_frac<<<grid_for(count, 256), 256, 0, st>>>((double*)x, (double*)p, (const double*)psi[0],
                                                        (const double*)psi[1], (const double*)psi[2], lognp, D / box,
                                                        pfac);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- second-order LPT
// With Psi1 = -grad phi1, phi1_ij = -d_j Psi1_i, and the 2LPT source
//   S = sum_{i<j} (phi1_ii phi1_jj - phi1_ij^2)
// (Bouchet et al. 1995; Scoccimarro 1998) is gathered over the three components:
//   stage 0 (Psi1_x): S = -(d_y Psi_x)^2 - (d_z Psi_x)^2,   A = d_x Psi_x
//   stage 1 (Psi1_y): S += A d_y Psi_y - (d_z Psi_y)^2,      A += d_y Psi_y
//   stage 2 (Psi1_z): S += A d_z Psi_z
template <typename T>
__global__ void k_lpt2_source(int stage, const T* __restrict__ d0, const T* __restrict__ d1, const T* __restrict__ d2,
                              T* __restrict__ s, T* __restrict__ a, int64_t count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (stage == 0) {
            const T y = d1[i], z = d2[i];
            s[i] = -(y * y) - z * z;
            a[i] = d0[i];
        } else if (stage == 1) {
            const T y = d1[i], z = d2[i], ai = a[i];
            s[i] += ai * y - z * z;
            a[i] = ai + y;
        } else {
            s[i] += a[i] * d2[i];
        }
    }
}

cudaError_t lpt2_source(int stage, void* const* d, void* s, void* a, int64_t count, int precision, cudaStream_t st) {
    if (precision == PM_FP32_FIXED)
        k_lpt2_source<float><<<grid_for(count, 256), 256, 0, st>>>(stage, (const float*)d[0], (const float*)d[1],
                                                                   (const float*)d[2], (float*)s, (float*)a, count);
    else
        k_lpt2_source<double><<<grid_for(count, 256), 256, 0, st>>>(stage, (const double*)d[0], (const double*)d[1],
                                                                    (const double*)d[2], (double*)s, (double*)a, count);
    return cudaGetLastError();
}

// x = q + D1 Psi1 + D2 Psi2, p = pfac1 Psi1 + pfac2 Psi2.  Psi1 may live in p: each thread
// reads the three components of its particle before writing them (no __restrict__ there).
struct Psi3 {
    const void* c[3];
};

__global__ void k_ic2_ticks(uint32_t* __restrict__ x, float* p, Psi3 ps1, Psi3 ps2, int lognp, TickScale disp1,
                            TickScale disp2, df pfac1, df pfac2) {
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int sh = 32 - lognp;
    const int mask = (1 << lognp) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t q[3] = {(uint32_t)((i >> (2 * lognp)) & mask) << sh, (uint32_t)((i >> lognp) & mask) << sh,
                               (uint32_t)(i & mask) << sh};
        float a1[3], a2[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            a1[j] = ((const float*)ps1.c[j])[i];
            a2[j] = ((const float*)ps2.c[j])[i];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            x[j * count + i] = q[j] + disp_ticks(a1[j], disp1, a2[j], disp2);
            p[j * count + i] = round_df(a1[j] * pfac1 + a2[j] * pfac2);
        }
    }
}

__global__ void k_ic2_frac(double* __restrict__ x, double* p, Psi3 ps1, Psi3 ps2, int lognp, double disp1,
                           double disp2, double pfac1, double pfac2) {
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int mask = (1 << lognp) - 1;
    const double inv_np = ldexp(1.0, -lognp);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double q[3] = {(double)((i >> (2 * lognp)) & mask) * inv_np, (double)((i >> lognp) & mask) * inv_np,
                             (double)(i & mask) * inv_np};
        double a1[3], a2[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            a1[j] = ((const double*)ps1.c[j])[i];
            a2[j] = ((const double*)ps2.c[j])[i];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            double xj = q[j] + (disp1 * a1[j] + disp2 * a2[j]);
            xj -= floor(xj);
            x[j * count + i] = xj;
            p[j * count + i] = pfac1 * a1[j] + pfac2 * a2[j];
        }
    }
}

cudaError_t ic_place2(void* x, void* p, void* const* psi1, void* const* psi2, int np, int precision, double D1,
                      double D2, double pfac1, double pfac2, double box, cudaStream_t st) {
    const int lognp = ilog2(np);
    const int64_t count = (int64_t)np * np * np;
    const Psi3 a = {{psi1[0], psi1[1], psi1[2]}}, b = {{psi2[0], psi2[1], psi2[2]}};
    if (precision == PM_FP32_FIXED) {
        k_ic2_ticks<<<grid_for(count, 256), 256, 0, st>>>((uint32_t*)x, (float*)p, a, b, lognp,
                                                          tick_scale(D1 * 4294967296.0 / box),
                                                          tick_scale(D2 * 4294967296.0 / box), df_of(pfac1),
                                                          df_of(pfac2));
    } else {
        k_ic2_frac<<<grid_for(count, 256), 256, 0, st>>>((double*)x, (double*)p, a, b, lognp, D1 / box, D2 / box,
                                                         pfac1, pfac2);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- Philox phases
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two 32x32->64
// multiplies with the Philox multipliers, xor with the key, word permutation, and
// a Weyl-sequence key bump between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += W0;
            k1 += W1;
        }
        const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// Unit complex Gaussian of mode draw (r.x, r.y) by the Box-Muller transform: in FP64, and for
// FP32 phases in pairs of FP32 numbers (dfloat.cuh), which round to the same phases but for one in
// ten thousand (neighbouring FP32 numbers there).  At 512^3 the FP64 logarithm, square root and
// sine took 9.4 ms of the 16.5 ms of the initial conditions; this is bound by issue instead.
__device__ __forceinline__ void unit_gaussian(uint4 r, double2& g) {
    const double u1 = ((double)r.x + 0.5) * 2.3283064365386963e-10;  // 2^-32
    const double u2 = ((double)r.y + 0.5) * 2.3283064365386963e-10;
    const double amp = sqrt(-log(u1));
    double s, c;
    sincospi(2.0 * u2, &s, &c);
    g = make_double2(amp * c, amp * s);
}
__device__ __forceinline__ void unit_gaussian(uint4 r, float2& g) {
    const df amp = df_sqrt(neg_log_unit(r.x));
    df s, c;
    sincos_unit(r.y, s, c);
    g = make_float2(round_df(amp * c), round_df(amp * s));
}

// Unit complex Gaussian per wavevector on the [kz][kx][ky] half grid; Hermitian
// partners on kz = 0 are conjugates of the canonical draw; Nyquist and zero modes 0.
// blockIdx.y selects the field of a batch, drawn from seeds.s[field].
struct Seeds {
    static constexpr int MAX = 128;
    uint64_t s[MAX];
};
template <typename T>
__global__ void k_noise(cplx<T>* __restrict__ spec, int logn, Seeds seeds) {
    const int n = 1 << logn, M = n >> 1;
    const uint32_t total = (uint32_t)(M + 1) << (2 * logn);  // at most 513 x 2^20
    const uint64_t seed = seeds.s[blockIdx.y];
    spec += (size_t)blockIdx.y * total;
    const uint32_t seed_lo = (uint32_t)seed, seed_hi = (uint32_t)(seed >> 32);
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int nz = (int)(e >> (2 * logn));
        const int nx = signed_k((int)(e >> logn) & (n - 1), n), ny = signed_k((int)e & (n - 1), n);
        cplx<T> g;
        g.x = T(0);
        g.y = T(0);
        const bool nyq = (2 * nx == -n) || (2 * ny == -n) || (nz == M);
        if (!nyq && (nx | ny | nz) != 0) {
            const bool canonical = nz > 0 || ny > 0 || (ny == 0 && nx > 0);
            const int cx = canonical ? nx : -nx, cy = canonical ? ny : -ny;
            const uint4 r = philox4x32_10(make_uint4((uint32_t)cx, (uint32_t)cy, (uint32_t)nz, 0u), seed_lo, seed_hi);
            unit_gaussian(r, g);
            if (!canonical) g.y = -g.y;
        }
        spec[e] = g;
    }
}

template <typename T>
cudaError_t noise(cplx<T>* spec, int n, const uint64_t* seeds, int nfields, cudaStream_t st) {
    const int64_t total = (int64_t)(n / 2 + 1) * n * n;
    for (int f0 = 0; f0 < nfields; f0 += Seeds::MAX) {
        const int c = nfields - f0 < Seeds::MAX ? nfields - f0 : Seeds::MAX;
        Seeds s = {};
        for (int i = 0; i < c; ++i) s.s[i] = seeds[f0 + i];
        k_noise<T><<<dim3(grid_for(total, 256), c), 256, 0, st>>>(spec + (size_t)f0 * total, ilog2(n), s);
    }
    return cudaGetLastError();
}
template cudaError_t noise<float>(float2*, int, const uint64_t*, int, cudaStream_t);
template cudaError_t noise<double>(double2*, int, const uint64_t*, int, cudaStream_t);

// The FP32 phases of pairs of Philox words, by themselves.
__global__ void k_phase_check(const uint2* __restrict__ words, int64_t count, float2* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const uint2 w = words[i];
        float2 g;
        unit_gaussian(make_uint4(w.x, w.y, 0u, 0u), g);
        out[i] = g;
    }
}
cudaError_t phase_check(const uint32_t* words, int64_t count, float* out, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    k_phase_check<<<grid_for(count, 256), 256, 0, st>>>((const uint2*)words, count, (float2*)out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- GR displacement combination
// xi = x_GR - x_N on the coarse lattice (exact minimum image on ticks), trilinear in
// the Lagrangian lattice index to the target lattice (r = npt / npc), x_t += xi.
__global__ void k_combine_ticks(uint32_t* __restrict__ xt, const uint32_t* __restrict__ xg,
                                const uint32_t* __restrict__ xn, int32_t* __restrict__ xi_out, int lognt,
                                int lognc) {
    const int64_t countt = (int64_t)1 << (3 * lognt);
    const int64_t countc = (int64_t)1 << (3 * lognc);
    const int logr = lognt - lognc;
    const int r = 1 << logr;
    const int maskt = (1 << lognt) - 1, maskc = (1 << lognc) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < countt;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int it[3] = {(int)((i >> (2 * lognt)) & maskt), (int)((i >> lognt) & maskt), (int)(i & maskt)};
        int base[3], off[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            base[j] = it[j] >> logr;
            off[j] = it[j] & (r - 1);
        }
        int64_t S[3] = {0, 0, 0};
#pragma unroll
        for (int dx = 0; dx < 2; ++dx)
#pragma unroll
            for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                for (int dz = 0; dz < 2; ++dz) {
                    const int64_t W = (int64_t)(dx ? off[0] : r - off[0]) * (dy ? off[1] : r - off[1]) *
                                      (dz ? off[2] : r - off[2]);
                    if (W == 0) continue;
                    const int64_t c = (((int64_t)((base[0] + dx) & maskc) << (2 * lognc)) |
                                       ((int64_t)((base[1] + dy) & maskc) << lognc) | ((base[2] + dz) & maskc));
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        const int32_t d = (int32_t)(xg[j * countc + c] - xn[j * countc + c]);
                        S[j] += W * (int64_t)d;
                    }
                }
        const int s = 3 * logr;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            int64_t q = S[j];
            if (s > 0) {  // round-half-even of S / 2^s
                const int64_t fl = S[j] >> s;
                const int64_t rem = S[j] - (fl << s);
                const int64_t half = (int64_t)1 << (s - 1);
                q = fl + ((rem > half || (rem == half && (fl & 1))) ? 1 : 0);
            }
            xt[j * countt + i] += (uint32_t)q;
            if (xi_out) xi_out[j * countt + i] = (int32_t)q;
        }
    }
}

// The same combination by blocks: one thread per coarse node b, for the r^3 targets whose
// lower coarse node is b (trilinear from the 8 nodes b + {0,1}^3; xi formed once per node).
// The r targets of a z-run sit together: their positions are read and written as one
// r-wide vector (r = 1, 2, 4), consecutive threads covering consecutive runs.
template <int LOGR>
__global__ void __launch_bounds__(256) k_combine_blocks(uint32_t* __restrict__ xt, const uint32_t* __restrict__ xg,
                                                        const uint32_t* __restrict__ xn, int32_t* __restrict__ xi_out,
                                                        int lognc) {
    constexpr int r = 1 << LOGR, s = 3 * LOGR;
    typedef typename std::conditional<r == 4, uint4, typename std::conditional<r == 2, uint2, uint32_t>::type>::type V;
    const int maskc = (1 << lognc) - 1, lognt = lognc + LOGR;
    const int64_t countc = (int64_t)1 << (3 * lognc), countt = (int64_t)1 << (3 * lognt);
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < countc;
         b += (int64_t)gridDim.x * blockDim.x) {
        const int bx = (int)(b >> (2 * lognc)), by = (int)((b >> lognc) & maskc), bz = (int)(b & maskc);
        int32_t xi[3][8];  // corner q = 4 dx + 2 dy + dz
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int64_t c = ((int64_t)((bx + (q >> 2)) & maskc) << (2 * lognc)) |
                              ((int64_t)((by + ((q >> 1) & 1)) & maskc) << lognc) | ((bz + (q & 1)) & maskc);
#pragma unroll
            for (int j = 0; j < 3; ++j) xi[j][q] = (int32_t)(xg[j * countc + c] - xn[j * countc + c]);
        }
        // one x plane of the r^3 target block at a time: its r x 3 target vectors are loaded
        // before any arithmetic, so their latencies overlap instead of forming r^2 x 3 chains
#pragma unroll(r <= 2 ? 2 : 1)
        for (int ox = 0; ox < r; ++ox) {
            V v[r][3];
#pragma unroll
            for (int oy = 0; oy < r; ++oy) {
                const int64_t t0 = ((((int64_t)(r * bx + ox) << lognt) + (r * by + oy)) << lognt) + r * bz;
#pragma unroll
                for (int j = 0; j < 3; ++j) v[oy][j] = *reinterpret_cast<const V*>(xt + j * countt + t0);
            }
#pragma unroll
            for (int oy = 0; oy < r; ++oy) {
                const int64_t t0 = ((((int64_t)(r * bx + ox) << lognt) + (r * by + oy)) << lognt) + r * bz;
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    uint32_t add[r];
#pragma unroll
                    for (int oz = 0; oz < r; ++oz) {
                        // S = sum over the corners of (weights in units of 1/r per axis) xi; exact in 64 bits
                        int64_t S = 0;
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const int wx = (q >> 2) ? ox : r - ox, wy = ((q >> 1) & 1) ? oy : r - oy,
                                      wz = (q & 1) ? oz : r - oz;
                            S += (int64_t)xi[j][q] * (wx * wy * wz);
                        }
                        int64_t qv = S;
                        if (s > 0) {  // round-half-even of S / r^3
                            const int64_t fl = S >> s;
                            const int64_t rem = S - (fl << s);
                            const int64_t half = (int64_t)1 << (s > 0 ? s - 1 : 0);
                            qv = fl + ((rem > half || (rem == half && (fl & 1))) ? 1 : 0);
                        }
                        add[oz] = (uint32_t)qv;
                    }
                    uint32_t* vv = reinterpret_cast<uint32_t*>(&v[oy][j]);
#pragma unroll
                    for (int oz = 0; oz < r; ++oz) vv[oz] += add[oz];
                    *reinterpret_cast<V*>(xt + j * countt + t0) = v[oy][j];
                    if (xi_out) {
                        V w;
                        uint32_t* ww = reinterpret_cast<uint32_t*>(&w);
#pragma unroll
                        for (int oz = 0; oz < r; ++oz) ww[oz] = add[oz];
                        *reinterpret_cast<V*>(xi_out + j * countt + t0) = w;
                    }
                }
            }
        }
    }
}

__global__ void k_combine_frac(double* __restrict__ xt, const double* __restrict__ xg, const double* __restrict__ xn,
                               double* __restrict__ xi_out, int lognt, int lognc) {
    const int64_t countt = (int64_t)1 << (3 * lognt);
    const int64_t countc = (int64_t)1 << (3 * lognc);
    const int logr = lognt - lognc;
    const int r = 1 << logr;
    const double inv_r3 = ldexp(1.0, -3 * logr);
    const int maskt = (1 << lognt) - 1, maskc = (1 << lognc) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < countt;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int it[3] = {(int)((i >> (2 * lognt)) & maskt), (int)((i >> lognt) & maskt), (int)(i & maskt)};
        int base[3], off[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            base[j] = it[j] >> logr;
            off[j] = it[j] & (r - 1);
        }
        double S[3] = {0, 0, 0};
        for (int dx = 0; dx < 2; ++dx)
            for (int dy = 0; dy < 2; ++dy)
                for (int dz = 0; dz < 2; ++dz) {
                    const int W = (dx ? off[0] : r - off[0]) * (dy ? off[1] : r - off[1]) * (dz ? off[2] : r - off[2]);
                    if (W == 0) continue;
                    const int64_t c = (((int64_t)((base[0] + dx) & maskc) << (2 * lognc)) |
                                       ((int64_t)((base[1] + dy) & maskc) << lognc) | ((base[2] + dz) & maskc));
                    for (int j = 0; j < 3; ++j) {
                        double d = xg[j * countc + c] - xn[j * countc + c];
                        d -= rint(d);
                        S[j] += (double)W * d;
                    }
                }
        for (int j = 0; j < 3; ++j) {
            const double xi = S[j] * inv_r3;
            double xj = xt[j * countt + i] + xi;
            xj -= floor(xj);
            xt[j * countt + i] = xj;
            if (xi_out) xi_out[j * countt + i] = xi;
        }
    }
}

cudaError_t combine(void* xt, const void* xg, const void* xn, void* xi_out, int npt, int npc, int precision,
                    cudaStream_t st) {
    const int lognt = ilog2(npt), lognc = ilog2(npc);
    const int64_t count = (int64_t)npt * npt * npt;
    const int64_t countc = (int64_t)npc * npc * npc;
    // vector accesses need 4 r-byte alignment (the library's particle arrays are 256-byte aligned)
    const bool aligned = (uintptr_t)xt % 16 == 0 && (uintptr_t)xi_out % 16 == 0;
    if (precision == PM_FP32_FIXED && aligned && lognt - lognc <= 2) {
        const unsigned g = grid_for(countc, 256);
        if (lognt == lognc)
            k_combine_blocks<0><<<g, 256, 0, st>>>((uint32_t*)xt, (const uint32_t*)xg, (const uint32_t*)xn,
                                                   (int32_t*)xi_out, lognc);
        else if (lognt == lognc + 1)
            k_combine_blocks<1><<<g, 256, 0, st>>>((uint32_t*)xt, (const uint32_t*)xg, (const uint32_t*)xn,
                                                   (int32_t*)xi_out, lognc);
        else
            k_combine_blocks<2><<<g, 256, 0, st>>>((uint32_t*)xt, (const uint32_t*)xg, (const uint32_t*)xn,
                                                   (int32_t*)xi_out, lognc);
    } else if (precision == PM_FP32_FIXED)
        k_combine_ticks<<<grid_for(count, 256), 256, 0, st>>>((uint32_t*)xt, (const uint32_t*)xg,
                                                              (const uint32_t*)xn, (int32_t*)xi_out, lognt, lognc);
    else
        k_combine_frac<<<grid_for(count, 256), 256, 0, st>>>((double*)xt, (const double*)xg, (const double*)xn,
                                                             (double*)xi_out, lognt, lognc);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- fill
template <typename T>
__global__ void k_fill(T* __restrict__ a, int64_t count, T v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = v;
}
cudaError_t fill(void* a, int64_t count, int precision, double v, cudaStream_t st) {
    if (precision == PM_FP32_FIXED)
        k_fill<float><<<grid_for(count, 256), 256, 0, st>>>((float*)a, count, (float)v);
    else
        k_fill<double><<<grid_for(count, 256), 256, 0, st>>>((double*)a, count, v);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- Lagrangian displacement
// d = x - q (minimum image) in Mpc/h for the np^3 lattice-ordered particles, q the node of
// particle id = (ix np + iy) np + iz.  Ticks: the uint32 difference read as int32 is the
// minimum image exactly.
__global__ void k_disp_ticks(const uint32_t* __restrict__ x, float* __restrict__ d, int lognp, float tick_mpc) {
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int mask = (1 << lognp) - 1;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t q[3] = {(uint32_t)((i >> (2 * lognp)) & mask) << (32 - lognp),
                               (uint32_t)((i >> lognp) & mask) << (32 - lognp), (uint32_t)(i & mask) << (32 - lognp)};
#pragma unroll
        for (int j = 0; j < 3; ++j) d[j * count + i] = (float)(int32_t)(x[j * count + i] - q[j]) * tick_mpc;
    }
}
__device__ __noinline__ double minus_rint(double x) { return x - rint(x); }
__global__ void k_disp_frac(const double* __restrict__ x, double* __restrict__ d, int lognp, double box) {
    const int64_t count = (int64_t)1 << (3 * lognp);
    const int mask = (1 << lognp) - 1;
    const double inv_np = 1.0 / (double)(1 << lognp);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const int q[3] = {(int)((i >> (2 * lognp)) & mask), (int)((i >> lognp) & mask), (int)(i & mask)};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // the nearest image is only looked for beyond half the box
            double v = fma((double)q[j], -inv_np, x[j * count + i]);  // q inv_np is exact
            if (!(((unsigned)__double2hiint(v) & 0x7fffffffu) < 0x3fe00000u)) v = minus_rint(v);
            d[j * count + i] = v * box;
        }
    }
}
cudaError_t lagrangian_displacement(const void* x, void* d, int np, int precision, double box, cudaStream_t st) {
    const int lognp = ilog2(np);
    const int64_t count = (int64_t)np * np * np;
    if (precision == PM_FP32_FIXED)
        k_disp_ticks<<<grid_for(count, 256), 256, 0, st>>>((const uint32_t*)x, (float*)d, lognp,
                                                           (float)(box / 4294967296.0));
    else
        k_disp_frac<<<grid_for(count, 256), 256, 0, st>>>((const double*)x, (double*)d, lognp, box);
    return cudaGetLastError();
}

// Positions in Mpc/h in [0, L): uint32 ticks times L / 2^32 (exact in double, then rounded
// down to float, so that no position rounds up to L), or box fractions times L.
__global__ void k_pos_ticks(const uint32_t* __restrict__ x, float* __restrict__ out, int64_t n, double tick_mpc) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __double2float_rd((double)x[i] * tick_mpc);
}
__global__ void k_pos_frac(const double* __restrict__ x, double* __restrict__ out, int64_t n, double box) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = x[i] * box;
}
cudaError_t positions_mpc(const void* x, void* out, int64_t count, int precision, double box, cudaStream_t st) {
    const int64_t n = 3 * count;
    if (n == 0) return cudaSuccess;
    if (precision == PM_FP32_FIXED)
        k_pos_ticks<<<grid_for(n, 256), 256, 0, st>>>((const uint32_t*)x, (float*)out, n, box / 4294967296.0);
    else
        k_pos_frac<<<grid_for(n, 256), 256, 0, st>>>((const double*)x, (double*)out, n, box);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- position check
// Counts FP64 box-fraction positions that are not finite or lie outside [0, 1) (one
// warp-aggregated atomic a warp).
__global__ void k_count_outside(const double* __restrict__ x, int64_t count, unsigned long long* __restrict__ bad) {
    unsigned long long mine = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        // 0 <= v < 1 on the bits (not the FP64 pipe): -0 passes, NaN does not
        const unsigned long long v = __double_as_longlong(x[i]);
        mine += ((unsigned)(v >> 32) < 0x3ff00000u || (v << 1) == 0) ? 0ull : 1ull;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(bad, mine);
}
cudaError_t count_outside_box(const double* x, int64_t count, unsigned long long* bad, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess || count == 0) return e;
    k_count_outside<<<grid_for(count, 256), 256, 0, st>>>(x, count, bad);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- cell keys and stable order
__global__ void k_cell_keys(const void* __restrict__ xv, int64_t count, int precision, int logn, float inv_cell_ticks,
                            uint32_t* __restrict__ keys, uint32_t* __restrict__ counts) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        int b[3];
        if (precision == PM_FP32_FIXED) {
            const uint32_t* x = (const uint32_t*)xv;
            for (int j = 0; j < 3; ++j) b[j] = cic_ticks(x[j * count + i], logn, inv_cell_ticks).i0;
        } else {
            const double* x = (const double*)xv;
            for (int j = 0; j < 3; ++j) b[j] = cic_frac(x[j * count + i], logn).i0;
        }
        const uint32_t key = ((uint32_t)b[0] << (2 * logn)) | ((uint32_t)b[1] << logn) | (uint32_t)b[2];
        keys[i] = key;
        if (counts) atomicAdd(&counts[key], 1u);
    }
}

// Exclusive scan, 4 elements per thread, 1024 threads per block.
__global__ void __launch_bounds__(1024) k_scan_block(const uint32_t* __restrict__ in, uint32_t* __restrict__ out,
                                                     int64_t count, uint32_t* __restrict__ block_sums) {
    __shared__ uint32_t warp_tot[32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * 4096 + 4 * tid;
    uint32_t v[4];
    uint32_t local = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = (base + k < count) ? in[base + k] : 0u;
        const uint32_t t = v[k];
        v[k] = local;
        local += t;
    }
    uint32_t incl = local;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        uint32_t w = warp_tot[lane];
        uint32_t wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, d);
            if (lane >= d) wi += y;
        }
        warp_tot[lane] = wi - w;  // exclusive warp offsets
        if (lane == 31 && block_sums) block_sums[blockIdx.x] = wi;
    }
    __syncthreads();
    const uint32_t off = warp_tot[wid] + (incl - local);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (base + k < count) out[base + k] = v[k] + off;
}

__global__ void k_scan_add(uint32_t* __restrict__ out, int64_t count, const uint32_t* __restrict__ sums) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] += sums[i / 4096];
}

// Exclusive scan of count uint32 values; scratch: scan_scratch_words(count) words.
static int64_t scan_scratch_words(int64_t count) {
    int64_t words = 0;
    while (count > 4096) {
        count = (count + 4095) / 4096;
        words += count + 1;
    }
    return words + 1;
}
static cudaError_t scan_u32(const uint32_t* in, uint32_t* out, int64_t count, uint32_t* scratch, cudaStream_t st) {
    const int64_t nblk = (count + 4095) / 4096;
    if (nblk <= 1) {
        k_scan_block<<<1, 1024, 0, st>>>(in, out, count, nullptr);
        return cudaGetLastError();
    }
    uint32_t* sums = scratch;
    k_scan_block<<<(unsigned)nblk, 1024, 0, st>>>(in, out, count, sums);
    cudaError_t e = scan_u32(sums, sums, nblk, scratch + nblk + 1, st);
    if (e != cudaSuccess) return e;
    k_scan_add<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(out, count, sums);
    return cudaGetLastError();
}

cudaError_t scan_exclusive_u32(const uint32_t* in, uint32_t* out, int64_t count, void* scratch, cudaStream_t st) {
    return scan_u32(in, out, count, (uint32_t*)scratch, st);
}

size_t scan_scratch_bytes(int64_t count) { return sizeof(uint32_t) * (size_t)(scan_scratch_words(count) + 64); }

__global__ void k_scatter_unstable(const uint32_t* __restrict__ keys, int64_t count, uint32_t* __restrict__ cursor,
                                   uint32_t* __restrict__ order) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        order[atomicAdd(&cursor[keys[i]], 1u)] = (uint32_t)i;
}

// Sorts at most MAX distinct ids: loaded together, each placed by the number of smaller ones.
template <uint32_t MAX>
__device__ __forceinline__ void sort_in_registers(uint32_t* a, uint32_t len) {
    uint32_t v[MAX];
#pragma unroll
    for (uint32_t k = 0; k < MAX; ++k) v[k] = k < len ? a[k] : 0xffffffffu;
#pragma unroll
    for (uint32_t k = 0; k < MAX; ++k) {
        uint32_t rank = 0;
#pragma unroll
        for (uint32_t m = 0; m < MAX; ++m) rank += v[m] < v[k] ? 1u : 0u;
        if (k < len) a[rank] = v[k];
    }
}

// Within each cell the ids were placed in arbitrary order; sort them ascending (up to MAX in
// registers, longer buckets by Shell sort with gaps 1, 4, 13, ...), which makes the whole order
// stable in id.  A mesh whose cells all run at once is bound by its longest buckets, MAX = 16 (32^3
// cells, 300,000 points, the whole sort: 55 us, 59 with 8 and with Shell sorts alone); on finer ones the
// walk over the cells, most of them empty or short, counts, and MAX = 8 keeps its registers at 32
// (256^3 cells, 1000 points: 166 us as without the register sorts, 177 with 16).
template <uint32_t MAX>
__global__ void __launch_bounds__(256)
    k_sort_buckets(const uint32_t* __restrict__ start, const uint32_t* __restrict__ cursor, int64_t ncell,
                   uint32_t* __restrict__ order) {
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t s = start[c], e = cursor[c];
        const uint32_t len = e - s;
        if (len < 2) continue;
        uint32_t* a = order + s;
        if (len <= 4) {
            sort_in_registers<4>(a, len);
            continue;
        }
        if (len <= 8) {
            sort_in_registers<8>(a, len);
            continue;
        }
        if (MAX > 8 && len <= MAX) {
            sort_in_registers<MAX>(a, len);
            continue;
        }
        uint32_t gap = 1;
        while (gap < len / 3) gap = 3 * gap + 1;
        for (; gap > 0; gap /= 3)
            for (uint32_t i = gap; i < len; ++i) {
                const uint32_t v = a[i];
                uint32_t j = i;
                while (j >= gap && a[j - gap] > v) {
                    a[j] = a[j - gap];
                    j -= gap;
                }
                a[j] = v;
            }
    }
}

size_t cell_sort_scratch_bytes(int64_t count, int n) {
    const int64_t ncell = (int64_t)n * n * n;
    (void)count;
    return sizeof(uint32_t) * (size_t)(3 * ncell + scan_scratch_words(ncell) + 64);
}

cudaError_t cell_sort(const void* x, int64_t count, int precision, int n, uint32_t* keys, uint32_t* order,
                      void* scratch, cudaStream_t st) {
    const int logn = ilog2(n);
    const int64_t ncell = (int64_t)n * n * n;
    uint32_t* counts = (uint32_t*)scratch;
    uint32_t* start = counts + ncell;
    uint32_t* cursor = start + ncell;
    uint32_t* sc = cursor + ncell;
    const float inv = (float)ldexp(1.0, -(32 - logn));
    cudaError_t e;
    if (order) {
        e = cudaMemsetAsync(counts, 0, sizeof(uint32_t) * ncell, st);
        if (e != cudaSuccess) return e;
    }
    if (count > 0)
        k_cell_keys<<<grid_for(count, 256), 256, 0, st>>>(x, count, precision, logn, inv, keys,
                                                          order ? counts : nullptr);
    e = cudaGetLastError();
    if (e != cudaSuccess || !order) return e;
    e = scan_u32(counts, start, ncell, sc, st);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(cursor, start, sizeof(uint32_t) * ncell, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    if (count > 0) k_scatter_unstable<<<grid_for(count, 256), 256, 0, st>>>(keys, count, cursor, order);
    const auto sort = ncell <= 2048 * (int64_t)num_sms() ? k_sort_buckets<16> : k_sort_buckets<8>;
    sort<<<grid_for(ncell, 256), 256, 0, st>>>(start, cursor, ncell, order);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- cell order without caller scratch
// Counting scratch for cell_sort_static: a fixed device array that every call on this
// GPU shares (it lives until the process exits).  Host code must not use the symbol
// as an address: the device address is looked up once per device below.
constexpr int64_t kStaticSortCells = (int64_t)64 * 64 * 64;
constexpr int64_t kStaticSortWords = 3 * kStaticSortCells + 4096;
static __device__ __align__(256) uint32_t g_sort_scratch[kStaticSortWords];

static std::mutex g_sort_mutex;
struct StaticSortAddr {
    unsigned long long ctx_id = 0;  // CUDA context the address belongs to (0: none yet)
    uint32_t* ptr = nullptr;
};
static StaticSortAddr g_sort_addr[128];

int64_t cell_sort_static_max_cells() { return kStaticSortCells; }

// Unique id of the calling thread's current CUDA context (0 when there is none), from the
// driver's cuCtxGetCurrent / cuCtxGetId reached through the runtime's entry-point query.
static unsigned long long current_context_id() {
    typedef int (*GetCurrent)(void**);
    typedef int (*GetId)(void*, unsigned long long*);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    if (!get_current || !get_id) {
        void* f1 = nullptr;
        void* f2 = nullptr;
        cudaDriverEntryPointQueryResult q1, q2;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) != cudaSuccess ||
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) != cudaSuccess ||
            q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return 0;
        }
        get_current = (GetCurrent)f1;
        get_id = (GetId)f2;
    }
    void* ctx = nullptr;
    unsigned long long id = 0;
    if (get_current(&ctx) != 0 || !ctx || get_id(ctx, &id) != 0) return 0;
    return id;
}

// Device address of g_sort_scratch in the current device's current context.  It is looked
// up (cudaGetSymbolAddress) on the first call in each context and cached under the
// context's id, so a context that is torn down and made again (cudaDeviceReset, a new
// primary context) gets a fresh lookup instead of a stale address.
static cudaError_t static_sort_scratch(uint32_t** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_sort_mutex);
    StaticSortAddr& a = g_sort_addr[dev];
    unsigned long long id = current_context_id();
    if (id == 0 || id != a.ctx_id || !a.ptr) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_sort_scratch);  // makes the runtime's context current if needed
        if (e != cudaSuccess) return e;
        if (id == 0) id = current_context_id();
        a.ctx_id = id;
        a.ptr = (uint32_t*)p;
    }
    *out = a.ptr;
    return cudaSuccess;
}

cudaError_t cell_sort_static(const void* x, int64_t count, int precision, int n, uint32_t* keys, uint32_t* order,
                             cudaStream_t st) {
    uint32_t* scratch = nullptr;
    cudaError_t e = static_sort_scratch(&scratch);
    if (e != cudaSuccess) return e;
    // cell_sort clears the counts it needs before use, so stale contents of the
    // shared array from an earlier call do not leak into this one
    return cell_sort(x, count, precision, n, keys, order, scratch, st);
}

}  // namespace pm

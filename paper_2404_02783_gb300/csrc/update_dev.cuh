// Device pieces of the particle update shared by particles.cu and update.cu: the CIC
// decode of uint32 tick positions, the per-particle gather + kick + drift, and the
// fixed-point deposit tile of a Lagrangian block of particles.
#pragma once

#include <stdint.h>

#include "internal.h"
#include "pm_common.cuh"

namespace pm {

// ---------------------------------------------------------------- CIC decode
struct CicF {
    int i0, i1;
    float w1;
};
__device__ __forceinline__ CicF cic_ticks(uint32_t u, int logn, float inv_cell_ticks) {
    const int sh = 32 - logn;
    const uint32_t t = u - (1u << (sh - 1));
    CicF c;
    c.i0 = (int)(t >> sh);
    c.i1 = (c.i0 + 1) & ((1 << logn) - 1);
    c.w1 = __uint2float_rn(t & ((1u << sh) - 1u)) * inv_cell_ticks;
    return c;
}
// Deposit of lattice-ordered particles (count = np^3, id = (ix np + iy) np + iz) by
// Lagrangian tiles.  A block of lattice sites, 16 x 16 x 32 mesh cells' worth (R = n / np cells per
// lattice step), has the particles that have not travelled far in that mesh box widened by H cells
// on every side, which a CTA accumulates in shared memory and then adds to the global mesh once
// per cell.  A particle whose CIC stencil leaves the box adds its weights to global memory
// directly, so the result is the same CIC density for any displacement.  A CTA owns TX x TY x TZ
// sites, the whole block or (XC of its 16 cells in x, tile_depth) a slice of it where blocks would
// leave SMs without one.  A slice keeps the block's box: with H cells around the slice's own
// instead, clumped particles added one by one in FP32, and a 64^3 lattice collapsed block by block
// had an error of 9.1e-7 for 2.7e-8.
//
// The tile accumulates in fixed point: each weight is rounded to a multiple of 2^-24
// (half a quantum at most, 3e-8, below the FP32 rounding of a sum near 1) and added
// with a native 32-bit integer atomic (shared-memory float atomics are a compare-and-
// swap loop on this part), so the tile sum is exact and independent of the order of the
// additions as long as no cell reaches 256 mass units.  The additions return nothing and test
// nothing; instead the sum of all cells is compared with the sum of all additions, both in 64
// bits, before the tile is flushed: each wrap of a 32-bit cell takes exactly 2^32 from the
// former.  In a tile that fails the comparison (a cell of 256 times the mean density) the words
// are the cells' totals modulo 2^32 and go to the mesh as such; the particles are added again from
// the positions just written, in steps of 2^12 quanta, which gives the wraps (tile_wraps), and a
// cell's h wraps, 256 h mass units, are added to the mesh at once.
// The box starts HZ = 4 cells below the tile in z so that its rows are made of 16-byte
// chunks aligned in the mesh: the flush adds four cells per vector reduction.
template <int R, int XC = 16>
struct DepTile {
    static constexpr int THREADS = 512;
    static constexpr int TX = XC / R, TY = 16 / R, TZ = 32 / R, H = 2, HZ = 4;
    static constexpr int DX = 16 + 2 * H, DY = TY * R + 2 * H, DZ = TZ * R + 2 * HZ;
    static constexpr int CELLS = DX * DY * DZ, CZ = DZ / 4, PLANE = DY * CZ;  // 16-byte chunks a row, an x plane
    static constexpr int PER = TX * TY * TZ;
    static constexpr bool SLICE = XC < 16;
    // x of the box's first cell for the tile bx along x
    static __device__ __forceinline__ int box_x(int bx) { return (bx * TX * R & ~15) - H; }
    static constexpr int PLANES = THREADS / PLANE;     // x planes a pass over the chunks takes at once
    static_assert(TX >= 1 && PER * R * R * R <= 8192, "tile mass bound");
    static_assert(DZ % 4 == 0 && (TZ * R) % 4 == 0 && HZ % 4 == 0, "z box made of aligned 16-byte chunks");
    static_assert(CELLS % 4 == 0 && PLANES >= 1, "whole vectors");
};

__device__ __forceinline__ void red_add_v4(float* dst, float4 v) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"l"(dst), "f"(v.x), "f"(v.y),
                 "f"(v.z), "f"(v.w)
                 : "memory");
}

constexpr float kTileQuanta = 16777216.0f;  // 2^24 quanta per unit mass
constexpr float kTileQuantum = 5.9604644775390625e-08f;  // 2^-24

// What a thread adds to its tile: the sum of its additions (at most 64 mass units, 2^30: one
// particle of four cells a lattice step) and, in a slice, the x planes that they fall in, since a
// slice fills few of its box's and the rest need not be read when it ends.
struct TileAdds {
    uint32_t sum = 0;
    int first = 1 << 20, last = -1;
    template <class D>
    __device__ __forceinline__ void reach(int dx) {
        if constexpr (D::SLICE) first = min(first, dx), last = max(last, dx + 1);
    }
};

// Adds w quanta to a cell and to the thread's sum.
__device__ __forceinline__ void tile_add(uint32_t* lo, int c, float w, TileAdds& t) {
    const uint32_t v = __float2uint_rn(w);
    atomicAdd(lo + c, v);
    t.sum += v;
}
// The second accumulation of a tile counts in steps of 2^kCoarse quanta.  A cell of total T, made
// of N <= 8192 additions, then holds S with T - S 2^12 in [0, N 2^12), at most 2^25, widened by the
// few quanta an addition by which the sweeps' merged weights may round apart from the particles'
// own.  The first accumulation's word is T mod 2^32; with its top bit the number of wraps,
// floor(T / 2^32) <= 32, is that of S 2^12 - top 2^31 + 2^30, which stays 2^29 clear of either end.
constexpr int kCoarse = 12;
__device__ __forceinline__ float tile_wraps(uint32_t S, unsigned top) {
    return 256.0f * (float)(((int)S - (int)(top << (31 - kCoarse)) + (1 << (30 - kCoarse))) >> (32 - kCoarse));
}

template <int WORDS>
__device__ __forceinline__ void tile_zero(uint32_t* words) {
    for (int c = threadIdx.x; c < WORDS / 4; c += blockDim.x)
        reinterpret_cast<uint4*>(words)[c] = make_uint4(0u, 0u, 0u, 0u);
}

// One particle's CIC weights into the tile (box origin o*) or, outside it, into rho.  quanta =
// mass 2^24 (a power of two times the mass: the weights are the same numbers, scaled).
// AGAIN: the second accumulation of a tile, of the particles inside the box alone.
template <class D, bool AGAIN>
__device__ __forceinline__ void tile_deposit(uint32_t* lo, float* __restrict__ rho, uint32_t u0,
                                             uint32_t u1, uint32_t u2, int logn, float inv_cell_ticks, int ox,
                                             int oy, int oz, float quanta, TileAdds& t) {
    const int nm = (1 << logn) - 1;
    const CicF cx = cic_ticks(u0, logn, inv_cell_ticks);
    const CicF cy = cic_ticks(u1, logn, inv_cell_ticks);
    const CicF cz = cic_ticks(u2, logn, inv_cell_ticks);
    const float wx[2] = {1.0f - cx.w1, cx.w1}, wy[2] = {1.0f - cy.w1, cy.w1}, wz[2] = {1.0f - cz.w1, cz.w1};
    const int dx = (cx.i0 - ox) & nm, dy = (cy.i0 - oy) & nm, dz = (cz.i0 - oz) & nm;
    if (dx < D::DX - 1 && dy < D::DY - 1 && dz < D::DZ - 1) {
        const int c0 = (dx * D::DY + dy) * D::DZ + dz;
        if (!AGAIN) t.reach<D>(dx);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const float wab = quanta * wx[a] * wy[b];
                const int c = c0 + (a * D::DY + b) * D::DZ;
                if (AGAIN) {
                    atomicAdd(lo + c, __float2uint_rn(wab * wz[0]) >> kCoarse);
                    atomicAdd(lo + c + 1, __float2uint_rn(wab * wz[1]) >> kCoarse);
                } else {
                    tile_add(lo, c, wab * wz[0], t);
                    tile_add(lo, c + 1, wab * wz[1], t);
                }
            }
    } else if (!AGAIN) {
        const uint32_t ix[2] = {(uint32_t)cx.i0, (uint32_t)cx.i1}, iy[2] = {(uint32_t)cy.i0, (uint32_t)cy.i1};
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const float wab = quanta * kTileQuantum * wx[a] * wy[b];
                float* row = rho + (((ix[a] << logn) + iy[b]) << logn);
                atomicAdd(row + cz.i0, wab * wz[0]);
                atomicAdd(row + cz.i1, wab * wz[1]);
            }
    }
}

// f(chunk, lx, ly, lz4) for every 16-byte chunk of the tile's planes first..last: a thread keeps its
// place in the x plane and walks the planes, so nothing is divided per chunk.
template <class D, class F>
__device__ __forceinline__ void for_chunks(int first, int last, F f) {
    const int lz4 = threadIdx.x % D::CZ, ly = (threadIdx.x / D::CZ) % D::DY, l0 = threadIdx.x / D::PLANE;
    if (l0 >= D::PLANES) return;
#pragma unroll 2
    for (int lx = first + l0; lx <= last; lx += D::PLANES) f((lx * D::DY + ly) * D::CZ + lz4, lx, ly, lz4);
}

// Mesh cell of the first of the tile's chunk (lx, ly, lz4); box origin o*, oz a multiple of 4.
__device__ __forceinline__ uint32_t chunk_cell(int lx, int ly, int lz4, int ox, int oy, int oz, int logn) {
    const int nm = (1 << logn) - 1;
    return ((((uint32_t)((ox + lx) & nm) << logn) + (uint32_t)((oy + ly) & nm)) << logn) + ((oz + 4 * lz4) & nm);
}

// Adds the cells of the tile's planes first..last to rho (16-byte aligned), four z-cells per
// reduction.
template <class D>
__device__ __forceinline__ void tile_flush(const uint32_t* lo, float* __restrict__ rho, int ox, int oy, int oz,
                                           int logn, int first, int last) {
    for_chunks<D>(first, last, [&](int c, int lx, int ly, int lz4) {
        const uint4 l = reinterpret_cast<const uint4*>(lo)[c];
        if (l.x | l.y | l.z | l.w)
            red_add_v4(rho + chunk_cell(lx, ly, lz4, ox, oy, oz, logn),
                       make_float4(__uint2float_rn(l.x) * kTileQuantum, __uint2float_rn(l.y) * kTileQuantum,
                                   __uint2float_rn(l.z) * kTileQuantum, __uint2float_rn(l.w) * kTileQuantum));
    });
}

// Ends a tile in which cells passed 2^32 quanta: the words are added to rho, their top bits kept
// (four a chunk; a thread has at most DX / PLANES of them), the tile is accumulated again in coarse
// steps (add() deposits the thread's particles from their written positions with AGAIN) and the
// wraps are added.
template <class D, class F>
__device__ __forceinline__ void tile_again(uint32_t* lo, float* __restrict__ rho, int ox, int oy, int oz, int logn,
                                           F add) {
    static_assert(4 * ((D::DX + D::PLANES - 1) / D::PLANES) <= 64, "top bits of a thread's chunks");
    tile_flush<D>(lo, rho, ox, oy, oz, logn, 0, D::DX - 1);
    unsigned long long tops = 0;
    for_chunks<D>(0, D::DX - 1, [&](int c, int, int, int) {
        const uint4 l = reinterpret_cast<const uint4*>(lo)[c];
        tops = tops << 4 | (l.x >> 31) << 3 | (l.y >> 31) << 2 | (l.z >> 31) << 1 | l.w >> 31;
        reinterpret_cast<uint4*>(lo)[c] = make_uint4(0u, 0u, 0u, 0u);
    });
    __syncthreads();
    add();
    __syncthreads();
    int left = 0;  // chunks of the thread that follow
    for_chunks<D>(0, D::DX - 1, [&](int, int, int, int) { ++left; });
    for_chunks<D>(0, D::DX - 1, [&](int c, int lx, int ly, int lz4) {
        const uint4 s = reinterpret_cast<const uint4*>(lo)[c];
        const unsigned t = (unsigned)(tops >> (4 * --left));
        const float4 v = make_float4(tile_wraps(s.x, t >> 3 & 1u), tile_wraps(s.y, t >> 2 & 1u),
                                     tile_wraps(s.z, t >> 1 & 1u), tile_wraps(s.w, t & 1u));
        if (v.x + v.y + v.z + v.w > 0.0f) red_add_v4(rho + chunk_cell(lx, ly, lz4, ox, oy, oz, logn), v);
    });
}

// Ends a tile: compares the sum of its cells with the sum of all additions (`adds` of every
// thread) and flushes it, or calls again(), which ends in tile_again, when they differ.  Every
// thread of the CTA calls it.
template <class D, class F>
__device__ __forceinline__ void tile_close(uint32_t* lo, float* __restrict__ rho, int ox, int oy, int oz, int logn,
                                           const TileAdds& adds, F again) {
    __shared__ unsigned long long missing;
    __shared__ int span[2];
    if (threadIdx.x == 0) {
        missing = 0;
        span[0] = D::DX, span[1] = -1;
    }
    __syncthreads();
    int first = 0, last = D::DX - 1;
    if constexpr (D::SLICE) {
        const int a = __reduce_min_sync(0xffffffffu, adds.first), b = __reduce_max_sync(0xffffffffu, adds.last);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&span[0], a);
            atomicMax(&span[1], b);
        }
        __syncthreads();
        first = span[0], last = span[1];
    }
    unsigned long long d = adds.sum;
    for_chunks<D>(first, last, [&](int c, int, int, int) {
        const uint4 l = reinterpret_cast<const uint4*>(lo)[c];
        d -= (unsigned long long)l.x + l.y + l.z + l.w;
    });
    // the warp's sum of d modulo 2^64 in three limbs
    const uint32_t l0 = __reduce_add_sync(0xffffffffu, (uint32_t)d & 0xffffu);
    const uint32_t l1 = __reduce_add_sync(0xffffffffu, (uint32_t)d >> 16);
    const uint32_t l2 = __reduce_add_sync(0xffffffffu, (uint32_t)(d >> 32));
    if ((threadIdx.x & 31) == 0)
        atomicAdd(&missing, (unsigned long long)l0 + ((unsigned long long)l1 << 16) + ((unsigned long long)l2 << 32));
    __syncthreads();
    if (missing == 0) tile_flush<D>(lo, rho, ox, oy, oz, logn, first, last);
    else again();
}

// Deposit of a thread walking its lattice row along x (R = 1).  The next particle usually
// sits one cell further in x with the same y and z cells; its lower-x CIC corners are then
// this particle's upper-x corners, so the upper-plane weights are carried (W, for the cell
// dnext) and added with the next particle's lower plane: 4 tile atomics a particle instead
// of 8.  A particle whose stencil leaves the box adds to rho directly.
struct SweepCarry {
    int dnext = -1;  // tile cell of the carried plane's (b, c) = (0, 0) corner, -1: none
    float W[4];      // carried weights, corner (b, c) = 2 b + c
    TileAdds adds;
};

template <class D>
__device__ __forceinline__ void sweep_carried(uint32_t* lo, SweepCarry& sc) {
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) tile_add(lo, sc.dnext + b * D::DZ + c, sc.W[2 * b + c], sc.adds);
}

template <class D>
__device__ __forceinline__ void sweep_deposit(uint32_t* lo, float* __restrict__ rho, uint32_t u0, uint32_t u1,
                                              uint32_t u2, int logn, float inv_cell_ticks, int ox, int oy, int oz,
                                              float quanta, SweepCarry& sc) {
    const int nm = (1 << logn) - 1;
    const CicF cx = cic_ticks(u0, logn, inv_cell_ticks);
    const CicF cy = cic_ticks(u1, logn, inv_cell_ticks);
    const CicF cz = cic_ticks(u2, logn, inv_cell_ticks);
    const float wy[2] = {1.0f - cy.w1, cy.w1}, wz[2] = {1.0f - cz.w1, cz.w1};
    const float m0 = quanta * (1.0f - cx.w1), m1 = quanta * cx.w1;
    const int dx = (cx.i0 - ox) & nm, dy = (cy.i0 - oy) & nm, dz = (cz.i0 - oz) & nm;
    if (dx < D::DX - 1 && dy < D::DY - 1 && dz < D::DZ - 1) {
        const int c0 = (dx * D::DY + dy) * D::DZ + dz;
        sc.adds.reach<D>(dx);
        float w0[4];
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int c = 0; c < 2; ++c) w0[2 * b + c] = m0 * wy[b] * wz[c];
        if (c0 == sc.dnext) {
#pragma unroll
            for (int q = 0; q < 4; ++q) w0[q] += sc.W[q];
        } else if (sc.dnext >= 0) {
            sweep_carried<D>(lo, sc);
        }
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                tile_add(lo, c0 + b * D::DZ + c, w0[2 * b + c], sc.adds);
                sc.W[2 * b + c] = m1 * wy[b] * wz[c];
            }
        sc.dnext = c0 + D::DY * D::DZ;
    } else {
        if (sc.dnext >= 0) sweep_carried<D>(lo, sc);
        sc.dnext = -1;
        const uint32_t ix[2] = {(uint32_t)cx.i0, (uint32_t)cx.i1}, iy[2] = {(uint32_t)cy.i0, (uint32_t)cy.i1};
        const float mx[2] = {m0 * kTileQuantum, m1 * kTileQuantum};
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                float* row = rho + (((ix[a] << logn) + iy[b]) << logn);
                atomicAdd(row + cz.i0, mx[a] * wy[b] * wz[0]);
                atomicAdd(row + cz.i1, mx[a] * wy[b] * wz[1]);
            }
    }
}

// ---------------------------------------------------------------- interp + kick + drift
// First-order gradient (PM_GRAD_FD1): the force -grad of the CIC interpolant of the
// potential inside the particle's cell, from its eight corners: L[q] on the lower x plane,
// U[q] on the upper one, corner (b, c) = 2 b + c for (y, z); inv_d = nmesh / L.
//   g_x = inv_d sum_bc wy_b wz_c (L - U)
//   g_y = inv_d sum_c wz_c [wx0 (L_0c - L_1c) + wx1 (U_0c - U_1c)]
//   g_z = inv_d sum_b wy_b [wx0 (L_b0 - L_b1) + wx1 (U_b0 - U_b1)]
template <typename T>
__device__ __forceinline__ void fd1_force(const T* L, const T* U, T wx0, T wx1, const T* wy, const T* wz, T inv_d,
                                          T& f0, T& f1, T& f2) {
    T gx = T(0), gy = T(0), gz = T(0);
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) gx += wy[b] * wz[c] * (L[2 * b + c] - U[2 * b + c]);
#pragma unroll
    for (int c = 0; c < 2; ++c) gy += wz[c] * (wx0 * (L[c] - L[2 + c]) + wx1 * (U[c] - U[2 + c]));
#pragma unroll
    for (int b = 0; b < 2; ++b) gz += wy[b] * (wx0 * (L[2 * b] - L[2 * b + 1]) + wx1 * (U[2 * b] - U[2 * b + 1]));
    f0 = inv_d * gx;
    f1 = inv_d * gy;
    f2 = inv_d * gz;
}

// The CIC corners of one x plane of a mesh of ROWS z rows a cell row: 32-bit element offsets
// (3 n^3 < 2^32) of (y, z) corner q = 2 b + c, the periodic wrap included.  One offset serves
// the three components of the force meshes (kForceRows), a row apart.
template <int ROWS>
struct PlaneCorners {
    uint32_t o00;
    int dy, dz;
    __device__ __forceinline__ PlaneCorners(int ix, const CicF& cy, const CicF& cz, int logn)
        : o00((uint32_t)((((ix << logn) + cy.i0) * ROWS) << logn) + (uint32_t)cz.i0),
          dy((cy.i1 - cy.i0) * (ROWS << logn)), dz(cz.i1 - cz.i0) {}
    __device__ __forceinline__ uint32_t operator[](int q) const {
        return o00 + (uint32_t)((q & 2 ? dy : 0) + (q & 1 ? dz : 0));
    }
};

// p += kick * g(x);  x += drift * p   (g = -grad phi gathered with the deposit's weights; the
// force meshes in the layout kForceRows).  FD: g is the potential, a plain mesh, differentiated
// to first order (fd1_force).
template <bool FD>
__device__ __forceinline__ void ikd_particle(uint32_t& u0, uint32_t& u1, uint32_t& u2, float& p0, float& p1,
                                             float& p2, int logn, float inv_cell_ticks, const float* g,
                                             float kick, float drift_ticks, float inv_d) {
    constexpr int ROWS = FD ? 1 : kForceRows;
    const CicF cx = cic_ticks(u0, logn, inv_cell_ticks);
    const CicF cy = cic_ticks(u1, logn, inv_cell_ticks);
    const CicF cz = cic_ticks(u2, logn, inv_cell_ticks);
    const float wx[2] = {1.0f - cx.w1, cx.w1}, wy[2] = {1.0f - cy.w1, cy.w1}, wz[2] = {1.0f - cz.w1, cz.w1};
    const PlaneCorners<ROWS> k[2] = {{cx.i0, cy, cz, logn}, {cx.i1, cy, cz, logn}};
    float f0 = 0.f, f1 = 0.f, f2 = 0.f;
    if constexpr (FD) {
        float P[2][4];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int q = 0; q < 4; ++q) P[a][q] = g[k[a][q]];
        fd1_force<float>(P[0], P[1], wx[0], wx[1], wy, wz, inv_d, f0, f1, f2);
    } else {
        const int n = 1 << logn;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const float* c0 = g + k[a][2 * b];
                const float* c1 = g + k[a][2 * b + 1];
                const float w0 = wx[a] * wy[b] * wz[0], w1 = wx[a] * wy[b] * wz[1];
                f0 = fmaf(w0, c0[0], fmaf(w1, c1[0], f0));
                f1 = fmaf(w0, c0[n], fmaf(w1, c1[n], f1));
                f2 = fmaf(w0, c0[2 * n], fmaf(w1, c1[2 * n], f2));
            }
    }
    p0 = fmaf(kick, f0, p0);
    p1 = fmaf(kick, f1, p1);
    p2 = fmaf(kick, f2, p2);
    // 32-bit conversion (the 64-bit one is several times slower here): exact for drifts under
    // half the box per step, i.e. |p drift_ticks| < 2^31, the range of any meaningful step
    u0 += (uint32_t)__float2int_rn(p0 * drift_ticks);
    u1 += (uint32_t)__float2int_rn(p1 * drift_ticks);
    u2 += (uint32_t)__float2int_rn(p2 * drift_ticks);
}

}  // namespace pm

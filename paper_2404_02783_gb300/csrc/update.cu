// The fused particle update of the FP32 PM step: CIC gather of the force at the old
// position, kick, drift, and the CIC deposit of the drifted position into the density of
// the next step, one pass over the lattice-ordered particles by Lagrangian tiles (KDK in a;
// counting density, Sec. 4).  Positions are uint32 ticks (2^32 per side).
#include "internal.h"
#include "particles.h"
#include "update_dev.cuh"

namespace pm {

// ---------------------------------------------------------------- kick + drift + next deposit
// One pass per step over the lattice-ordered particles by Lagrangian tiles: gather the
// force at x, kick, drift, and deposit the new position into the (zeroed) next
// density mesh through the tile's shared-memory accumulator, exactly as
// k_deposit_tiled would have done from the drifted positions.
// blockIdx.y selects the field of a batch of independent runs stored back to back
// (particles [field][3][np^3], force meshes [field][n][n][3][n], density [field][n^3]); scale =
// 2^32 / L of that field.  The mesh side 2^LOGN is a compile-time constant: the kernels were
// bound by issue without it, and its shifts, masks and row strides are then immediates.
template <int R, int XC, int LOGN, bool FD>
__global__ void __launch_bounds__(512, 2) k_ikd_deposit(const uint32_t* x, uint32_t* __restrict__ xo,
                                                        float* __restrict__ p, const float* g, float kick,
                                                        double drift, double scale0,
                                                        const double* __restrict__ scale_arr, float mass,
                                                        float* __restrict__ rho, float inv_d) {
    typedef DepTile<R, XC> D;
    constexpr int logn = LOGN, lognp = LOGN - (R == 4 ? 2 : R == 2 ? 1 : 0), np = 1 << lognp;
    constexpr int64_t count = (int64_t)1 << (3 * lognp);
    constexpr float inv_cell_ticks = 1.0f / (float)(1u << (32 - LOGN));
    extern __shared__ __align__(16) uint32_t lo[];  // D::CELLS
    {
        const int64_t fb = blockIdx.y;
        constexpr int64_t n3 = (int64_t)1 << (3 * LOGN);
        x += fb * 3 * count;
        xo += fb * 3 * count;
        p += fb * 3 * count;
        g += fb * (FD ? 1 : kForceRows) * n3;
        rho += fb * n3;
    }
    constexpr int ntz = np / D::TZ, nty = np / D::TY;
    const int bz = blockIdx.x % ntz, by = (blockIdx.x / ntz) % nty, bx = blockIdx.x / (ntz * nty);
    const int ox = D::box_x(bx), oy = by * D::TY * R - D::H, oz = bz * D::TZ * R - D::HZ;
    launch_next();
    tile_zero<D::CELLS>(lo);
    wait_previous();
    __syncthreads();
    const float drift_ticks = (float)(drift * (scale_arr ? scale_arr[blockIdx.y] : scale0));
    auto pid = [&](int e) -> int64_t {
        const int lz = e % D::TZ, ly = (e / D::TZ) % D::TY, lx = e / (D::TZ * D::TY);
        return ((((int64_t)(bx * D::TX + lx) << lognp) + by * D::TY + ly) << lognp) + bz * D::TZ + lz;
    };
    const float quanta = mass * kTileQuanta;
    TileAdds adds;
    // the next particle is loaded one iteration ahead (its latency overlaps this one's work)
    int64_t idn = pid(threadIdx.x);
    uint32_t nu0 = 0, nu1 = 0, nu2 = 0;
    float np0 = 0.f, np1 = 0.f, np2 = 0.f;
    if (D::PER >= 512 || threadIdx.x < D::PER) {
        nu0 = x[idn], nu1 = x[count + idn], nu2 = x[2 * count + idn];
        np0 = p[idn], np1 = p[count + idn], np2 = p[2 * count + idn];
    }
#pragma unroll 1
    for (int e = threadIdx.x; e < D::PER; e += 512) {
        const int64_t id = idn;
        uint32_t u0 = nu0, u1 = nu1, u2 = nu2;
        float p0 = np0, p1 = np1, p2 = np2;
        if (e + 512 < D::PER) {
            idn = pid(e + 512);
            nu0 = x[idn];
            nu1 = x[count + idn];
            nu2 = x[2 * count + idn];
            np0 = p[idn];
            np1 = p[count + idn];
            np2 = p[2 * count + idn];
        }
        ikd_particle<FD>(u0, u1, u2, p0, p1, p2, logn, inv_cell_ticks, g, kick, drift_ticks, inv_d);
        p[id] = p0;
        p[count + id] = p1;
        p[2 * count + id] = p2;
        xo[id] = u0;
        xo[count + id] = u1;
        xo[2 * count + id] = u2;
        tile_deposit<D, false>(lo, rho, u0, u1, u2, logn, inv_cell_ticks, ox, oy, oz, quanta, adds);
    }
    tile_close<D>(lo, rho, ox, oy, oz, logn, adds, [&] {
        tile_again<D>(lo, rho, ox, oy, oz, logn, [&] {
            for (int e = threadIdx.x; e < D::PER; e += 512) {
                const int64_t id = pid(e);
                tile_deposit<D, true>(lo, rho, xo[id], xo[count + id], xo[2 * count + id], logn, inv_cell_ticks, ox,
                                      oy, oz, quanta, adds);
            }
        });
    });
}

// The second accumulation of a sweep's tile (tile_close), from the thread's written positions.
template <int XC, int LOGN>
__device__ __forceinline__ void sweep_again(uint32_t* lo, const uint32_t* xo, float* rho, float quanta) {
    typedef DepTile<1, XC> D;
    constexpr int np = 1 << LOGN, ntz = np / D::TZ, nty = np / D::TY;
    constexpr int64_t count = (int64_t)1 << (3 * LOGN);
    const int bz = blockIdx.x % ntz, by = (blockIdx.x / ntz) % nty, bx = blockIdx.x / (ntz * nty);
    const int ox = D::box_x(bx), oy = by * D::TY - D::H, oz = bz * D::TZ - D::HZ;
    const int lz = threadIdx.x % D::TZ, ly = threadIdx.x / D::TZ;
    TileAdds adds;
    tile_again<D>(lo, rho, ox, oy, oz, LOGN, [&] {
        for (int lx = 0; lx < D::TX; ++lx) {
            const int64_t id = ((((int64_t)(bx * D::TX + lx) << LOGN) + by * D::TY + ly) << LOGN) + bz * D::TZ + lz;
            tile_deposit<D, true>(lo, rho, xo[id], xo[count + id], xo[2 * count + id], LOGN,
                                  1.0f / (float)(1u << (32 - LOGN)), ox, oy, oz, quanta, adds);
        }
    });
}
template <int XC, int LOGN>
__device__ __noinline__ void sweep_again_call(uint32_t* lo, const uint32_t* xo, float* rho, float quanta) {
    sweep_again<XC, LOGN>(lo, xo, rho, quanta);
}

// x and xo may be the same array (in-place update): every particle's position is read once,
// one iteration before its own thread writes it, and no thread touches another's particles.
// R = 1: each thread walks its lattice row along x (lx = 0..XC-1 at fixed ly, lz), so the
// next particle usually sits one cell further in x with the same y and z cells.  Then
// its lower-x CIC corners are this particle's upper-x corners: the gather keeps the 12
// upper-plane force values in registers and loads only the new plane, and the deposit
// carries the upper-plane weights in registers, adds them to the next particle's
// lower-plane weights and issues 4 tile atomics a particle instead of 8.  Any other
// particle takes the full path, so the result is the same CIC gather and deposit.
// Bound by the latency of the gather (256^3: long scoreboard 7.8 cycles an issue, issue 56% busy, 142 M
// warp instructions) with two CTAs an SM: the upper plane's loads, which every particle needs, are
// issued before the branch that reloads the lower plane (512^3, early and clustered steps: 1742 and
// 1953 us; after it 1826 and 2020).  The components are interpolated in packed pairs, and a tile
// without words for carries leaves the L1 cache 100 KB an SM instead of 68 for the force planes that
// neighbouring rows share (1733 and 1946 us with both the other way, 1723 and 1903 now; 2783 and 2633
// at 2 Mpc/h cells, where particles have moved furthest).  Holding the gather in flight across the
// previous particle's deposit spills at two 512-thread CTAs an SM (2293 us) and gains nothing at
// three 256-thread CTAs (1798 and 1958).
template <int XC, int LOGN, bool FD>
__global__ void __launch_bounds__(512, 2) k_ikd_deposit_sweep(const uint32_t* x, uint32_t* __restrict__ xo,
                                                              float* __restrict__ p, const float* g,
                                                              float kick, double drift, double scale0,
                                                              const double* __restrict__ scale_arr, float mass,
                                                              float* __restrict__ rho, float inv_d) {
    typedef DepTile<1, XC> D;
    static_assert(D::TY * D::TZ == 512, "one thread per (ly, lz); lx runs over the loop");
    constexpr int logn = LOGN, np = 1 << LOGN, NC = FD ? 1 : 3, ROWS = FD ? 1 : kForceRows;
    constexpr int64_t count = (int64_t)1 << (3 * LOGN);
    constexpr float inv_cell_ticks = 1.0f / (float)(1u << (32 - LOGN));
    extern __shared__ __align__(16) uint32_t lo[];  // D::CELLS
    {
        const int64_t fb = blockIdx.y;
        x += fb * 3 * count;
        xo += fb * 3 * count;
        p += fb * 3 * count;
        g += fb * ROWS * count;
        rho += fb * count;
    }
    constexpr int ntz = np / D::TZ, nty = np / D::TY;
    const int bz = blockIdx.x % ntz, by = (blockIdx.x / ntz) % nty, bx = blockIdx.x / (ntz * nty);
    const int ox = D::box_x(bx), oy = by * D::TY - D::H, oz = bz * D::TZ - D::HZ;
    launch_next();
    tile_zero<D::CELLS>(lo);
    wait_previous();
    __syncthreads();
    const float drift_ticks = (float)(drift * (scale_arr ? scale_arr[blockIdx.y] : scale0));
    const int lz = threadIdx.x % D::TZ, ly = threadIdx.x / D::TZ;
    const int64_t id0 = ((((int64_t)(bx * D::TX) << LOGN) + by * D::TY + ly) << LOGN) + bz * D::TZ + lz;
    constexpr int64_t xstride = (int64_t)1 << (2 * LOGN);
    uint32_t next_cell = 0xffffffffu;  // packed (ix, iy, iz) whose lower plane the registers hold
    float U[4][NC];                     // force (FD: potential) at the carried plane, corner (b, c) = 2 b + c
    const float quanta = mass * kTileQuanta;
    SweepCarry sc;                      // deposit weights carried to the next particle's plane
    // the next particle's position and momentum are loaded one iteration ahead, so their
    // memory latency overlaps the current particle's gather, update and deposit
    uint32_t nu0 = x[id0], nu1 = x[count + id0], nu2 = x[2 * count + id0];
    float np0 = p[id0], np1 = p[count + id0], np2 = p[2 * count + id0];
#pragma unroll 1
    for (int lx = 0; lx < D::TX; ++lx) {
        const int64_t id = id0 + lx * xstride;
        uint32_t u0 = nu0, u1 = nu1, u2 = nu2;
        float p0 = np0, p1 = np1, p2 = np2;
        if (lx + 1 < D::TX) {
            const int64_t idn = id + xstride;
            nu0 = x[idn];
            nu1 = x[count + idn];
            nu2 = x[2 * count + idn];
            np0 = p[idn];
            np1 = p[count + idn];
            np2 = p[2 * count + idn];
        }
        // ---- gather at the old position
        {
            const CicF cx = cic_ticks(u0, logn, inv_cell_ticks);
            const CicF cy = cic_ticks(u1, logn, inv_cell_ticks);
            const CicF cz = cic_ticks(u2, logn, inv_cell_ticks);
            const uint32_t yz = ((uint32_t)cy.i0 << LOGN) | (uint32_t)cz.i0;
            float L[4][NC];
            const bool same = (((uint32_t)cx.i0 << (2 * LOGN)) | yz) == next_cell;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < NC; ++j) L[q][j] = U[q][j];
            const PlaneCorners<ROWS> ku(cx.i1, cy, cz, logn);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < NC; ++j) U[q][j] = g[ku[q] + j * np];
            if (!same) {
                const PlaneCorners<ROWS> k(cx.i0, cy, cz, logn);
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int j = 0; j < NC; ++j) L[q][j] = g[k[q] + j * np];
            }
            next_cell = ((uint32_t)cx.i1 << (2 * LOGN)) | yz;
            const float wy[2] = {1.0f - cy.w1, cy.w1}, wz[2] = {1.0f - cz.w1, cz.w1};
            const float wx0 = 1.0f - cx.w1, wx1 = cx.w1;
            float f0 = 0.f, f1 = 0.f, f2 = 0.f;
            if constexpr (FD) {
                const float Lp[4] = {L[0][0], L[1][0], L[2][0], L[3][0]};
                const float Up[4] = {U[0][0], U[1][0], U[2][0], U[3][0]};
                fd1_force<float>(Lp, Up, wx0, wx1, wy, wz, inv_d, f0, f1, f2);
            } else {
                // along x and y on the corner pairs (b, 0), (b, 1), then along z
                float f[3];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const float2 t0 = fma2(wx1, make_float2(U[0][j], U[1][j]), mul2(wx0, make_float2(L[0][j], L[1][j])));
                    const float2 t1 = fma2(wx1, make_float2(U[2][j], U[3][j]), mul2(wx0, make_float2(L[2][j], L[3][j])));
                    const float2 t = fma2(wy[1], t1, mul2(wy[0], t0));
                    f[j] = fmaf(wz[0], t.x, wz[1] * t.y);
                }
                f0 = f[0], f1 = f[1], f2 = f[2];
            }
            p0 = fmaf(kick, f0, p0);
            p1 = fmaf(kick, f1, p1);
            p2 = fmaf(kick, f2, p2);
            u0 += (uint32_t)__float2int_rn(p0 * drift_ticks);
            u1 += (uint32_t)__float2int_rn(p1 * drift_ticks);
            u2 += (uint32_t)__float2int_rn(p2 * drift_ticks);
        }
        p[id] = p0;
        p[count + id] = p1;
        p[2 * count + id] = p2;
        xo[id] = u0;
        xo[count + id] = u1;
        xo[2 * count + id] = u2;
        // ---- deposit at the new position
        sweep_deposit<D>(lo, rho, u0, u1, u2, logn, inv_cell_ticks, ox, oy, oz, quanta, sc);
    }
    if (sc.dnext >= 0) sweep_carried<D>(lo, sc);  // the carried plane of the row's last particle
    tile_close<D>(lo, rho, ox, oy, oz, logn, sc.adds, [&] {
        // a call where the three components fill the registers (in line its values spill in the loop:
        // 1764 us against 1724); with the potential alone the call costs more (1680 us against 1501)
        if constexpr (FD) sweep_again<XC, LOGN>(lo, xo, rho, quanta);
        else sweep_again_call<XC, LOGN>(lo, xo, rho, quanta);
    });
}

namespace {

struct UpdateArgs {
    void* x;
    void* xo;
    void* p;
    const void* g;
    double kick, drift, scale0;
    const double* scale_arr;
    double mass;
    void* rho;
    double inv_d;
    int nfields;
    cudaStream_t st;
};

template <int R, int XC, int LOGN, bool FD>
cudaError_t ikd_launch(const UpdateArgs& a) {
    typedef DepTile<R, XC> D;
    constexpr int np = (1 << LOGN) / R;
    constexpr unsigned blocks = (unsigned)((np / D::TX) * (np / D::TY) * (np / D::TZ));
    const size_t smem = sizeof(uint32_t) * D::CELLS;
    const auto fn = [] {
        if constexpr (R == 1) return k_ikd_deposit_sweep<XC, LOGN, FD>;
        else return k_ikd_deposit<R, XC, LOGN, FD>;
    }();
    cudaError_t e = set_smem_once((const void*)fn, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(fn, dim3(blocks, a.nfields), 512, smem, a.st, true, (const uint32_t*)a.x, (uint32_t*)a.xo,
                          (float*)a.p, (const float*)a.g, (float)a.kick, a.drift, a.scale0, a.scale_arr, (float)a.mass,
                          (float*)a.rho, (float)a.inv_d);
}

// Meshes of 128^3 and up always fill the SMs with tiles of depth 16.
template <int R, bool FD>
cudaError_t ikd_sized(int n, int np, const UpdateArgs& a) {
    switch (n) {
        case 64:
            switch (tile_depth(R, np, a.nfields)) {
                case 2: return ikd_launch<R, R == 4 ? 4 : 2, 6, FD>(a);  // R = 4: a lattice step is four cells
                case 4: return ikd_launch<R, 4, 6, FD>(a);
                case 8: return ikd_launch<R, 8, 6, FD>(a);
                default: return ikd_launch<R, 16, 6, FD>(a);
            }
        case 128: return ikd_launch<R, 16, 7, FD>(a);
        case 256: return ikd_launch<R, 16, 8, FD>(a);
        case 512: return ikd_launch<R, 16, 9, FD>(a);
        case 1024: return ikd_launch<R, 16, 10, FD>(a);
        default: return cudaErrorInvalidValue;
    }
}

template <bool FD>
cudaError_t ikd_any(int n, int np, const UpdateArgs& a) {
    switch (n / np) {
        case 1: return ikd_sized<1, FD>(n, np, a);
        case 2: return ikd_sized<2, FD>(n, np, a);
        case 4: return ikd_sized<4, FD>(n, np, a);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Every slice of a block brings the block's box, so the deepest tile is used that still gives every SM
// one: 64^3 particles on 64^3 cells are 32 blocks, 256 slices of depth 2.  A step takes 24.4 us with
// those and 29.0 with 128 of depth 4; the update alone took 25.4 us with whole blocks and takes 10.6.
// From 152 blocks on whole ones are as good or better (64^3 on 128^3, 256 blocks: 15.0 us against 16.1
// and 18.5 at depths 8 and 4, with boxes of their own; 256^3: 237, 247, 269 us).
int tile_depth(int R, int np, int nfields) {
    const int64_t tiles = (int64_t)nfields * (np * R / 16) * (np * R / 16) * (np * R / 32);  // of depth 16
    return tiles >= num_sms() ? 16 : 2 * tiles >= num_sms() ? 8 : 4 * tiles >= num_sms() ? 4 : 2;
}

bool ikd_deposit_supported(int np, int precision, int n) {
    const int R = n / np;
    return precision == PM_FP32_FIXED && n >= 64 && (R == 1 || R == 2 || R == 4) && np >= 32 / R;
}

cudaError_t interp_kick_drift_deposit(void* x, void* p, int np, int precision, int n, const void* g, double kick,
                                      double drift, double box, double mass, void* rho, cudaStream_t st, int nfields,
                                      const double* scale_arr, void* x_out, double fd_inv_d) {
    if (!ikd_deposit_supported(np, precision, n) || nfields < 1 || (uintptr_t)rho % 16 != 0)
        return cudaErrorInvalidValue;
    const bool fd = fd_inv_d > 0.0;
    const UpdateArgs a{x, x_out ? x_out : x, p, g, kick, drift, 4294967296.0 / box, scale_arr, mass, rho,
                       fd ? fd_inv_d : 0.0, nfields, st};
    return fd ? ikd_any<true>(n, np, a) : ikd_any<false>(n, np, a);
}

}  // namespace pm

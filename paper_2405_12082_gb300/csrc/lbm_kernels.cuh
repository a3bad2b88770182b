// lbm_kernels.cuh -- kernels of the pipe-flow LBM, instantiated once per storage
// precision by lbm_f64.cu, lbm_f32.cu, lbm_f16s.cu and lbm_bf16.cu (each defines
// LBM_PREC before including this file).
#pragma once

#include <algorithm>
#include <type_traits>
#include <utility>

#include "lbm_internal.h"
#include "lbm_pair.cuh"

namespace lbm {

// ---- the fused step: load (stream) + wall + force + MRT collision + store ----------------
// One thread per fluid cell of every member (padding of the compact rows returns at once).  EXTRA selects
// what else the step does: EX_STATS adds u_z^k, k = 1..4, of the pre-collision state to
// the FP64 sums (sample steps); EX_MOMENTS stores rho, u and s4..s8 of the
// pre-collision state for the adjoint sweep.  BS threads per block, register budget
// for MINB resident blocks per SM.

// Whether the step's populations travel in storage units (the scaled half format with the
// default collision: the scale is applied inside collide, see there).
template <int P, int EXTRA, int MODEL>
__host__ __device__ constexpr bool raw_units() {
    return Storage<P>::kScaled && MODEL == MODEL_MRT_H6 && EXTRA != EX_MOMENTS;
}

// Force, collide and store one fluid cell p of member d whose 27 populations (f - w, or
// (f - w) 2^s in raw units) are in v.
template <int P, int PAR, int WALL, int EXTRA, int MODEL>
__device__ __forceinline__ void finish_cell(const StepArgs &a, const Member &d, const CellPos &p, int64_t t,
                                            typename Storage<P>::R stv, typename Storage<P>::R (&v)[Q]) {
    using R = typename Storage<P>::R;
    R gx, gy, gz;
    acceleration<R>(d, p, t, stv, gx, gy, gz);
    if constexpr (EXTRA == EX_MOMENTS) {
        R sk[5];
        const Macro<R> mm = collide<R>(v, gx, gy, gz, omega_of<R>(d), sk);
        R *mo = static_cast<R *>(a.moments) + p.lc;
        const int64_t n = d.scells;
        mo[0] = mm.rho;
        mo[n] = mm.ux;
        mo[2 * n] = mm.uy;
        mo[3 * n] = mm.uz;
#pragma unroll
        for (int k = 0; k < 5; ++k) mo[(4 + k) * n] = sk[k];
    } else {
        constexpr bool SC = Storage<P>::kScaled && MODEL == MODEL_MRT_H6;
        const Macro<R> mm = collide<R, MODEL, SC, P != LBM_F32>(v, gx, gy, gz, omega_of<R>(d), nullptr, lam1_of<R>(d),
                                                  (R)a.f16_inv, (R)a.f16_scale);
        if constexpr (EXTRA == EX_STATS) {
            const double uz = (double)mm.uz;
            add_stats(a.stats + d.doff + p.di, a.dstride, uz);
        }
    }
    if constexpr (P == LBM_F64) release_next_step();        // (see k_step)
    store_pops<P, PAR, WALL, raw_units<P, EXTRA, MODEL>()>(a, d, p, v);
}

// Stream, force, collide and store one fluid cell p of member d.
template <int P, int PAR, int WALL, int EXTRA, int MODEL>
__device__ __forceinline__ void step_cell(const StepArgs &a, const Member &d, const CellPos &p, int64_t t,
                                          typename Storage<P>::R stv) {
    using R = typename Storage<P>::R;
    R v[Q];
    load_pops<P, PAR, WALL, raw_units<P, EXTRA, MODEL>()>(a, d, p, v);
    finish_cell<P, PAR, WALL, EXTRA, MODEL>(a, d, p, t, stv, v);
}

// The cell above p (z + 1) in the same column: same in-plane data, one plane further.
__device__ __forceinline__ void next_plane(const Member &d, CellPos &p) {
    p.z += 1;
    p.lc += d.Ps;
    p.di += d.nx * d.ny;
    p.oz[0] = p.z == 0 ? (d.nz - 1) * d.Ps : -d.Ps;
    p.oz[2] = p.z == d.nz - 1 ? -(d.nz - 1) * d.Ps : d.Ps;
}

// ZC > 1: each thread takes ZC consecutive planes of one in-plane position (threads of a
// block stay consecutive in that position, so accesses stay coalesced); the position's
// table lookup and neighbour offsets are paid once per ZC cells.
template <int P, int PAR, int WALL, int EXTRA, int BS, int MINB, int MODEL = MODEL_MRT_H6, int ZC = 1>
__global__ void __launch_bounds__(BS, MINB) k_step(const __grid_constant__ StepArgs a) {
    using R = typename Storage<P>::R;
    // FP64 steps are bound by the FP64 units of each SM: a successor released at once packs its
    // blocks onto the SMs this grid leaves free (20 x 20 x 64 pipe: 31 us per step against 14.4
    // without overlap), so it is released before the stores, when the arithmetic is done
    if constexpr (P != LBM_F64) release_next_step();
    const int m = find_member(a, blockIdx.x);
    const Member &d = a.members[m];
    const uint32_t local = (uint32_t)(blockIdx.x - a.block0[m]) * BS + threadIdx.x;
    CellPos p;
    if (!cell_from_work(d, local, ZC, p)) return;
    const int64_t t = a.times ? a.times[a.tidx].t : a.t;
    const R stv = st_of<R>(a, m);
    await_previous_step();
#pragma unroll 1
    for (int k = 0; k < ZC; ++k) {
        if (k > 0) {
            if (p.z + 1 >= d.nz) break;
            next_plane(d, p);
        }
        step_cell<P, PAR, WALL, EXTRA, MODEL>(a, d, p, t, stv);
    }
}

// ---- software-pipelined persistent step (F32, F64 storage) -----------------------------------
// A persistent block walks over tiles of BS cells (grid-stride).  Before computing tile k
// each thread issues the 27 loads of its cell in tile k + 1 as cp.async copies into its
// own shared-memory column (stage (k+1) mod 2), so the loads of the next tile are in
// flight while the current one is computed, without holding registers.  Every AA slot is
// read and written by one cell only within a step, so prefetching ahead of other cells'
// stores is safe, and each thread reads back only what it copied itself: per-thread
// cp.async groups replace any block barrier.
__device__ __forceinline__ void cp_async_4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_8(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_one() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

extern __shared__ __align__(16) unsigned char lbm_smem[];

template <int P, int PAR, int WALL>
__device__ __forceinline__ void prefetch_pops(const StepArgs &a, const Member &d, const CellPos &p, uint32_t sbase,
                                              int stride_bytes) {
    using T = typename Storage<P>::T;
    const T *base = static_cast<const T *>(a.pops) + d.off;
    const uint32_t st = (uint32_t)a.stride;
    const uint32_t lc = (uint32_t)p.lc;
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int ib = opp_of(i);
        uint32_t idx;
        if constexpr (PAR == 0) {
            idx = i * st + lc;
        } else {
            const uint32_t pull = ib * st + (uint32_t)(p.lc + src_offset<i>(p));
            if constexpr (WALL == LBM_FULLWAY || (cx_of(i) == 0 && cy_of(i) == 0)) idx = pull;
            else idx = src_is_fluid<i>(p) ? pull : i * st + lc;
        }
        if constexpr (sizeof(T) == 8) cp_async_8(sbase + i * stride_bytes, base + idx);
        else cp_async_4(sbase + i * stride_bytes, base + idx);
    });
}

struct TileCell {
    int m;
    bool active;
    CellPos p;
};

template <int BS>
__device__ __forceinline__ TileCell tile_cell(const StepArgs &a, int tile) {
    TileCell c;
    c.m = 0;
    c.active = false;
    if (tile < a.nblocks_total) {
        c.m = find_member(a, tile);
        const Member &d = a.members[c.m];
        const uint32_t local = (uint32_t)(tile - a.block0[c.m]) * BS + threadIdx.x;
        // the grid covers the fluid columns of a dense pipe (make_args), else the stored cells
        if (d.fluidcol != nullptr) c.active = cell_from_work(d, local, 1, c.p);
        else if (local < (uint32_t)d.scells) c.active = cell_from_storage(d, local, c.p);
    }
    return c;
}

template <int P, int PAR, int WALL, int EXTRA, int BS, int MINB>
__global__ void __launch_bounds__(BS, MINB) k_step_pipe(const __grid_constant__ StepArgs a) {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(lbm_smem);
    const int stride_bytes = BS * (int)sizeof(T);            // one population column of a stage
    const uint32_t stage_bytes = (uint32_t)(Q * BS * sizeof(T));
    const uint32_t mine = smem0 + threadIdx.x * sizeof(T);
    const T *smem_t = reinterpret_cast<const T *>(lbm_smem) + threadIdx.x;
    int tile = blockIdx.x;
    TileCell cur = tile_cell<BS>(a, tile);
    if (cur.active) prefetch_pops<P, PAR, WALL>(a, a.members[cur.m], cur.p, mine, stride_bytes);
    cp_async_commit();
    const int64_t t = a.times ? a.times[a.tidx].t : a.t;
    for (int k = 0; tile < a.nblocks_total; ++k) {
        const int next_tile = tile + gridDim.x;
        TileCell nxt = tile_cell<BS>(a, next_tile);
        if (nxt.active)
            prefetch_pops<P, PAR, WALL>(a, a.members[nxt.m], nxt.p, mine + ((k + 1) & 1) * stage_bytes, stride_bytes);
        cp_async_commit();
        cp_async_wait_one();                                 // this thread's copies of tile k are done
        if (cur.active) {
            const Member &d = a.members[cur.m];
            const T *col = smem_t + (k & 1) * (Q * BS);
            R v[Q];
            const R inv = (R)a.f16_inv;
            sfor<0, Q>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                v[i] = S::ld(col + i * BS, inv);
            });
            if constexpr (WALL == LBM_BOUZIDI) bouzidi_load_fix<R>(d, cur.p, v);
            R gx, gy, gz;
            acceleration<R>(d, cur.p, t, st_of<R>(a, cur.m), gx, gy, gz);
            const Macro<R> mm = collide<R>(v, gx, gy, gz, omega_of<R>(d));
            if constexpr (EXTRA == EX_STATS) {
                const double uz = (double)mm.uz;
                add_stats(a.stats + d.doff + cur.p.di, a.dstride, uz);
            }
            store_pops<P, PAR, WALL>(a, d, cur.p, v);
        }
        tile = next_tile;
        cur = nxt;
    }
    cp_async_wait_all();
}

// ---- state I/O: the exact inverse of load_pops ---------------------------------------------
template <int P, int PAR, int WALL>
__device__ __forceinline__ void write_state(const StepArgs &a, const Member &d, const CellPos &p,
                                            typename Storage<P>::R (&v)[Q]) {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    T *base = static_cast<T *>(a.pops);
    const R sc = (R)a.f16_scale;
    if constexpr (WALL == LBM_BOUZIDI) {
        if (p.nb != 0x1FFu) {
            sfor<0, Q>([&](auto jc) {
                constexpr int j = decltype(jc)::value;
                if constexpr (cx_of(j) != 0 || cy_of(j) != 0) {
                    if (!dst_is_fluid<j>(p)) {
                        BLink<R> b = bouzidi_link<R, j>(d, p);
                        v[opp_of(j)] -= b.C * v[j];
                    }
                }
            });
        }
    }
    T *b = base + d.off;
    const uint32_t st = (uint32_t)a.stride;
    const uint32_t lc = (uint32_t)p.lc;
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int ib = opp_of(i);
        if constexpr (PAR == 0) {
            S::st(b + (i * st + lc), v[i], sc);
        } else {
            const uint32_t pull = ib * st + (uint32_t)(p.lc + src_offset<i>(p));
            if constexpr (WALL == LBM_FULLWAY || (cx_of(i) == 0 && cy_of(i) == 0)) {
                S::st(b + pull, v[i], sc);
            } else {
                const uint32_t own = i * st + lc;
                S::st(b + (src_is_fluid<i>(p) ? pull : own), v[i], sc);
            }
        }
    });
}

// Shifted second-order equilibrium f^eq(rho, u) - w (no force term).
template <class R>
__device__ __forceinline__ void feq_shifted_o2(R drho, R ux, R uy, R uz, R (&v)[Q]) {
    const R rho = R(1) + drho, uu = ux * ux + uy * uy + uz * uz;
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const R cu = cterm<cz_of(i)>(cterm<cy_of(i)>(cterm<cx_of(i)>(R(-0.0), ux), uy), uz);
        v[i] = R(w_of(i)) * (drho + rho * (R(3) * cu + R(4.5) * cu * cu - R(1.5) * uu));
    });
}

// Shifted equilibrium f^eq(rho, u) - w in the product form (no force term).
template <class R>
__device__ __forceinline__ void feq_shifted(R drho, R ux, R uy, R uz, R (&v)[Q]) {
    R dx[3], hx[3], dy[3], hy[3], dz[3], hz[3];
    axis_factors<R>(ux, R(0), dx, hx);
    axis_factors<R>(uy, R(0), dy, hy);
    axis_factors<R>(uz, R(0), dz, hz);
    const R rho = R(1) + drho;
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const R dxy = dx[cx_of(i) + 1] + dy[cy_of(i) + 1] + dx[cx_of(i) + 1] * dy[cy_of(i) + 1];
        const R pm1 = dxy + dz[cz_of(i) + 1] * (R(1) + dxy);
        v[i] = R(w_of(i)) * (drho + rho * pm1);
    });
}

template <int P, int PAR, int WALL>
__global__ void k_moments(const __grid_constant__ StepArgs a, int m, typename Storage<P>::R *rho,
                          typename Storage<P>::R *u) {
    using R = typename Storage<P>::R;
    const Member &d = a.members[m];
    const int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (local >= d.cells) return;
    CellPos p;
    if (!cell_from_dense(d, (uint32_t)local, p)) {
        rho[local] = 0;
        u[local] = 0;
        u[d.cells + local] = 0;
        u[2 * d.cells + local] = 0;
        return;
    }
    R v[Q];
    load_pops<P, PAR, WALL>(a, d, p, v);
    R gx, gy, gz;
    acceleration<R>(d, p, a.t, st_of<R>(a, m), gx, gy, gz);
    const Macro<R> mm = macroscopic<R>(v, gx, gy, gz);
    rho[local] = mm.rho;
    u[local] = mm.ux;
    u[d.cells + local] = mm.uy;
    u[2 * d.cells + local] = mm.uz;
}

template <int P, int PAR, int WALL>
__global__ void k_get_pops(const __grid_constant__ StepArgs a, int m, double *f) {
    using R = typename Storage<P>::R;
    const Member &d = a.members[m];
    const int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (local >= d.cells) return;
    CellPos p;
    const bool fluid = cell_from_dense(d, (uint32_t)local, p);
    R v[Q];
    if (fluid || WALL == LBM_FULLWAY) {
        load_pops<P, PAR, WALL>(a, d, p, v);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = 0;
    }
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        f[(int64_t)i * d.cells + local] = (double)v[i] + w_of(i);
    });
}

template <int P, int PAR, int WALL>
__global__ void k_set_pops(const __grid_constant__ StepArgs a, int m, const double *f) {
    using R = typename Storage<P>::R;
    const Member &d = a.members[m];
    const int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (local >= d.cells) return;
    CellPos p;
    if (!cell_from_dense(d, (uint32_t)local, p) && WALL != LBM_FULLWAY) return;
    R v[Q];
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        v[i] = (R)(f[(int64_t)i * d.cells + local] - w_of(i));
    });
    write_state<P, PAR, WALL>(a, d, p, v);
}

// ---- initial state ---------------------------------------------------------------------------
// SplitMix64 (Steele, Lea, Flood 2014): output n of seed s is mix64(s + (n+1) gamma).
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t n) {
    uint64_t z = seed + (n + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
// Box-Muller normal number (3 c + k) for cell c, component k.
__device__ __forceinline__ double normal_at(uint64_t seed, uint64_t cell, int k) {
    const uint64_t n1 = 2ull * (3ull * cell + (uint64_t)k);
    const double u1 = ((double)(splitmix64_at(seed, n1) >> 11) + 1.0) * 0x1.0p-53;
    const double u2 = (double)(splitmix64_at(seed, n1 + 1ull) >> 11) * 0x1.0p-53;
    return sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
}

template <int P, int WALL>
__global__ void k_init(const __grid_constant__ StepArgs a, int m, int profile, double noise_amp,
                       uint64_t seed, const double *rho_in, const double *u_in) {
    using R = typename Storage<P>::R;
    const Member &d = a.members[m];
    const int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (local >= d.cells) return;
    CellPos p;
    R v[Q];
    if (!cell_from_dense(d, (uint32_t)local, p)) {
        if (!d.compact) {                               // solid cells are stored only densely
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = 0;
            write_state<P, 0, LBM_FULLWAY>(a, d, p, v);   // plain own-slot write at t = 0
        }
        return;
    }
    double ux = 0, uy = 0, uz = 0, drho = 0;
    if (rho_in != nullptr) {
        drho = rho_in[local] - 1.0;
        ux = u_in[local];
        uy = u_in[d.cells + local];
        uz = u_in[2 * d.cells + local];
    } else {
        const double px = 0.5 * (double)(2 * p.x - d.nx + 1), py = 0.5 * (double)(2 * p.y - d.ny + 1);
        const double r = sqrt(px * px + py * py);
        const double nu = (1.0 / d.omega - 0.5) / 3.0;
        const double gz = d.g[2];
        if (profile == LBM_LAMINAR) {
            uz = gz * (d.R * d.R - r * r) / (4.0 * nu);
        } else if (profile == LBM_LOGLAW) {
            const double us = sqrt(gz * d.R / 2.0);
            const double dplus = (d.R - r) * us / nu;
            const double uplus = dplus <= 10.8 ? dplus : log(dplus) / 0.4 + 5.0;
            uz = us * uplus;
        }
        if (noise_amp != 0.0) {
            ux += noise_amp * normal_at(seed, (uint64_t)local, 0);
            uy += noise_amp * normal_at(seed, (uint64_t)local, 1);
            uz += noise_amp * normal_at(seed, (uint64_t)local, 2);
        }
    }
    if (a.collision & MODEL_O2) feq_shifted_o2<R>((R)drho, (R)ux, (R)uy, (R)uz, v);
    else feq_shifted<R>((R)drho, (R)ux, (R)uy, (R)uz, v);
    write_state<P, 0, WALL>(a, d, p, v);
}

// ---- reductions (deterministic two-pass) -------------------------------------------------------
template <int NV>
__device__ __forceinline__ void block_sum(double (&x)[NV], double *sh /* [NV][32] */) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_down_sync(0xFFFFFFFFu, x[k], o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k * 32 + warp] = x[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            x[k] = lane < nw ? sh[k * 32 + lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_down_sync(0xFFFFFFFFu, x[k], o);
        }
    }
}

// FP64 adds are what a sum of FP32 populations costs here (two lanes per SM and cycle: 81 adds
// and 27 conversions per cell took 10 ms on the R = 96 pipe, against 0.55 ms for reading it).
// So every thread keeps each population's sum over its cells as an unevaluated pair hi + lo of
// floats -- Knuth's two-sum: hi + x = s + e exactly -- where e joins lo by another two-sum, whose
// error (2^-48 of the magnitudes and less) goes to the thread's four sums r: nothing is lost but
// the rounding of r, and a thread's 27 pairs enter FP64 once, through the z-triplets of
// moment_sums.  (With lo's rounding dropped the pairs had to enter FP64 every eight cells and still
// lost up to 2^-45: fields, rings and sums of the R = 96 pipe 2,215 us, now 1,878.)  Cells with a
// value too large for FP32 sums (or not finite) are added in FP64.
__device__ __forceinline__ void add_sums(double (&acc)[5], const MomentSums<double> &m) {
    acc[0] += m.drho;
    acc[1] += m.jx;
    acc[2] += m.jy;
    acc[3] += m.jz;
}
// a + b = s + e exactly; returns s.
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}
template <int P, int PAR, int WALL>
__global__ void __launch_bounds__(REDUCE_BLOCK, 2) k_reduce(const __grid_constant__ StepArgs a, int m,
                                                         double *partials) {
    using R = typename Storage<P>::R;
    __shared__ double sh[5 * 32];
    const Member &d = a.members[m];
    double acc[5] = {0, 0, 0, 0, 0};
    float hi[Q], lo[Q], r[4] = {0.f, 0.f, 0.f, 0.f};      // r: mass, momentum
#pragma unroll
    for (int i = 0; i < Q; ++i) hi[i] = lo[i] = 0.f;
    const int64_t work = (int64_t)d.Pw * d.nz;
    for (int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; local < work;
         local += (int64_t)gridDim.x * blockDim.x) {
        CellPos p;
        if (cell_from_work(d, (uint32_t)local, 1, p)) {
            R v[Q];
            load_pops<P, PAR, WALL>(a, d, p, v);
            bool wide = false;
#pragma unroll
            for (int i = 0; i < Q; ++i) wide |= !(fabs(v[i]) < R(1e30));
            if (sizeof(R) == 8 || wide) {
                bool bad = false;
#pragma unroll
                for (int i = 0; i < Q; ++i) bad |= !isfinite(v[i]);
                acc[4] += bad ? 1.0 : 0.0;
            }
            if constexpr (sizeof(R) == 8) {
                add_sums(acc, moment_sums<double>(v));
            } else if (wide) {
                sfor<0, Q>([&](auto ic) {
                    constexpr int i = decltype(ic)::value, c[3] = {cx_of(i), cy_of(i), cz_of(i)};
                    const double x = (double)v[i];
                    acc[0] += x;
                    if constexpr (c[0] != 0) acc[1] += c[0] * x;
                    if constexpr (c[1] != 0) acc[2] += c[1] * x;
                    if constexpr (c[2] != 0) acc[3] += c[2] * x;
                });
            } else {
                sfor<0, 9>([&](auto kc) {                       // the z-triplet of column (cx, cy)
                    constexpr int cx = decltype(kc)::value % 3 - 1, cy = decltype(kc)::value / 3 - 1;
                    float q[3];
#pragma unroll
                    for (int z = 0; z < 3; ++z) {
                        const int i = dir_of(cx, cy, z - 1);
                        float e;
                        hi[i] = two_sum(hi[i], v[i], e);
                        lo[i] = two_sum(lo[i], e, q[z]);
                    }
                    const float s = __fadd_rn(__fadd_rn(q[0], q[1]), q[2]);
                    r[0] = __fadd_rn(r[0], s);
                    if constexpr (cx != 0) r[1] = __fmaf_rn((float)cx, s, r[1]);
                    if constexpr (cy != 0) r[2] = __fmaf_rn((float)cy, s, r[2]);
                    r[3] = __fadd_rn(r[3], __fsub_rn(q[2], q[0]));
                });
            }
        }
    }
    if constexpr (sizeof(R) == 4) {
        double x[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) x[i] = __dadd_rn((double)hi[i], (double)lo[i]);
        add_sums(acc, moment_sums<double>(x));
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += (double)r[k];
    }
    block_sum<5>(acc, sh);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 5; ++k) partials[blockIdx.x * 5 + k] = acc[k];
}

static __global__ void __launch_bounds__(REDUCE_BLOCK) k_reduce_final(const double *partials, int n, double *out) {
    __shared__ double sh[5 * 32];
    double acc[5] = {0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < n; b += blockDim.x)
#pragma unroll
        for (int k = 0; k < 5; ++k) acc[k] += partials[b * 5 + k];
    block_sum<5>(acc, sh);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 5; ++k) out[k] = acc[k];
}

// ---- coherent-structure rings, Sec. II.C -------------------------------------------------------
template <int P, int PAR, int WALL>
__device__ double uz_at(const StepArgs &a, const Member &d, int m, int x, int y, int z) {
    using R = typename Storage<P>::R;
    if (x < 0 || y < 0 || x >= d.nx || y >= d.ny) return 0.0;
    CellPos p;
    if (!cell_from_dense(d, (uint32_t)(((int64_t)z * d.ny + y) * d.nx + x), p)) return 0.0;
    R v[Q];
    load_pops<P, PAR, WALL>(a, d, p, v);
    R gx, gy, gz;
    acceleration<R>(d, p, a.t, st_of<R>(a, m), gx, gy, gz);
    return (double)macroscopic<R>(v, gx, gy, gz).uz;
}

// One block per (section, ring): bilinear samples of u_z into shared memory, then the
// DFT energies E_m = |sum_n u_n e^{-i m theta_n}|^2 / N^2 with warp-shuffle sums.  The N
// angles' sines and cosines (FP64: the slow units of this chip) are taken once per block, for
// the sample positions, and serve the DFT as its table: m n mod N, stepped without a division.
// R = 96 pipe, 3 rings x 16 sections of 1024 samples, m to 32: 0.076 ms (with a sine and a cosine
// per sample and mode one ring of 512 samples took 0.27 ms).
constexpr int MODES_BLOCK = 512;
template <int P, int PAR, int WALL>
__global__ void __launch_bounds__(MODES_BLOCK) k_modes(const __grid_constant__ StepArgs a, int m, const ModesArgs ma,
                                                       double *E) {
    extern __shared__ double smp[];            // [3][N]: u_z, cos, sin
    const Member &d = a.members[m];
    const int s = blockIdx.x / ma.n_rings, j = blockIdx.x % ma.n_rings;
    const int z = (int)(((int64_t)s * d.nz) / ma.n_sections);
    const int N = ma.n_theta;
    double *const cosn = smp + N, *const sinn = smp + 2 * N;
    const double xc = 0.5 * (d.nx - 1), yc = 0.5 * (d.ny - 1);
    const double r = ma.r_over_R[j] * d.R;
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        double sn, cs;
        sincospi(2.0 * (double)n / (double)N, &sn, &cs);
        cosn[n] = cs;
        sinn[n] = sn;
        const double px = xc + r * cs, py = yc + r * sn;
        const int i0 = (int)floor(px), j0 = (int)floor(py);
        const double fx = px - i0, fy = py - j0;
        const double u00 = uz_at<P, PAR, WALL>(a, d, m, i0, j0, z);
        const double u10 = uz_at<P, PAR, WALL>(a, d, m, i0 + 1, j0, z);
        const double u01 = uz_at<P, PAR, WALL>(a, d, m, i0, j0 + 1, z);
        const double u11 = uz_at<P, PAR, WALL>(a, d, m, i0 + 1, j0 + 1, z);
        smp[n] = (1 - fx) * (1 - fy) * u00 + fx * (1 - fy) * u10 + (1 - fx) * fy * u01 + fx * fy * u11;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int mode = warp; mode <= ma.n_modes; mode += nw) {
        double re = 0, im = 0;
        const int step = (int)(((int64_t)mode * 32) % N);
        int k = (int)(((int64_t)mode * lane) % N);          // mode n mod N
        for (int n = lane; n < N; n += 32) {
            re += smp[n] * cosn[k];
            im -= smp[n] * sinn[k];
            k += step;
            if (k >= N) k -= N;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            re += __shfl_down_sync(0xFFFFFFFFu, re, o);
            im += __shfl_down_sync(0xFFFFFFFFu, im, o);
        }
        if (lane == 0)
            E[((int64_t)s * ma.n_rings + j) * (ma.n_modes + 1) + mode] = (re * re + im * im) / ((double)N * N);
    }
}

// ---- trigger-force tables ---------------------------------------------------------------------
template <class R>
__global__ void k_force_tables(const Member *members, int m, R *ftab, R *ztab) {
    const Member &d = members[m];
    const int ncol = d.nx * d.ny;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < ncol) {
        double Px, Py, Pz;
        trigger_column(d, k % d.nx, k / d.nx, Px, Py, Pz);
        ftab[k] = (R)Px;
        ftab[ncol + k] = (R)Py;
        ftab[2 * ncol + k] = (R)Pz;
        if (d.compact && ((d.colmask[k] >> 4) & 1u)) {       // the same by stored position
            const int y = k / d.nx, x = k % d.nx;
            R *fc = static_cast<R *>(const_cast<void *>(d.ftabc)) + (d.rowbase[y] + x - d.rowx0[y]);
            fc[0] = (R)Px;
            fc[d.Ps] = (R)Py;
            fc[2 * (int64_t)d.Ps] = (R)Pz;
        }
    }
    if (k < d.nz) {
        double sz, cz;
        sincospi(2.0 * (double)d.kz * (double)k / (double)d.nz, &sz, &cz);
        ztab[k] = (R)cz;
        ztab[d.nz + k] = (R)sz;
    }
}

// ---- adjoint step ------------------------------------------------------------------------------
// Reverse of step t of a single half-way pipe.  mu = S^T lambda_{t+1} gathers
// lambda_i(x + c_i) when x + c_i is fluid and lambda_ibar(x) across a wall link (the
// transpose of half-way bounce-back; in AA terms, direction ibar's odd-step read); the
// wall-shear objective adds 2 c_iz / (T A_w) on wall links.  The collision is a function of
// rho, u and the raw shear moments m4..m8:
//   f*_j = w_j (rho P_j - 1) + (rho / 2) w_j g . grad_u P_j + (1 - omega) sum_k C_kj s_k,
//   P_j = psi(c_jx, u_x) psi(c_jy, u_y) psi(c_jz, u_z) (normalised), s_k = m_k - rho e_k(u)
//   + rho r_k(u, g) / 2,
// so lambda_t,i = A_rho + sum_a A_ua (c_ia - v_a) / rho + (1 - omega) sum_k q_k M_k(c_i)
// with v = u - g / 2, q_k = sum_j mu_j C_kj and A_rho, A_u the partial derivatives of
// sum_j mu_j f*_j.  The sums over j of mu_j w_j times products of psi and its first two
// u-derivatives are contracted axis by axis (z, then y, then x).  Per cell the FP64
// accumulators collect the objective, dJ/dg_z(x) and dJ/domega.
//
// One axis of a contraction, m the values at c = -1, 0, +1 (rest weight 4 times the others',
// the common 1/6 left to the end): with P = m+ + m-, D = m+ - m-, E = 2 P - 4 m0, S = P + 4 m0
//   sum psi m = S + 3 u (D + u E / 2),  sum psi' m = 3 (D + u E),  sum psi'' m = 3 E;
// f1 and f2 return the last two without their factor 3.
template <class R>
struct AxisSum { R f0, f1, f2; };
template <class R>
__device__ __forceinline__ AxisSum<R> axis_sum(R mm, R m0, R mp, R u3, R uh, R u) {
    const R P = add_(mp, mm), D = sub_(mp, mm);
    const R E = fma_(lit<R>(-4), m0, add_(P, P)), S = fma_(lit<R>(4), m0, P);
    return AxisSum<R>{fma_(u3, fma_(uh, E, D), S), fma_(u, E, D), E};
}

// One cell (R float or double, any plane) or the cells of planes z and z + 1 (R pf2, no
// periodic wrap between them) of position r: jterm, wterm their objective and dJ/domega terms.
// Bound by latency and issue (27 gathers, 9 moments, 27 stores per cell; L2 holds the fields of
// 50 MB each in part): pairs share the gather's addresses and halve the arithmetic's issue slots, and the
// axis sums above take 162 operations where psi, psi', psi'' products took 220.  R = 24 pipe,
// F32: 30 -> 26 us per step (128 threads x 4 blocks, 128 registers, no spills).
template <int P, int OBJ, class R>
__device__ __forceinline__ void adjoint_cells(const AdjArgs &j, const int4 ci, uint32_t r, int z, R &jterm, R &wterm) {
    using S = typename scalar_of<R>::type;
    constexpr bool TWO = std::is_same<R, pf2>::value;
    const AdjMember &d = j.one;
    const uint32_t ps = (uint32_t)d.Ps, nb = (uint32_t)ci.y, lc = r + (uint32_t)z * ps, n = d.n;
    auto ld = [&](const S *q, uint32_t k) -> R {
        if constexpr (TWO) return make_float2(q[k], q[k + ps]);
        else return q[k];
    };
    auto st = [&](S *q, uint32_t k, R v) {
        if constexpr (TWO) {
            q[k] = v.x;
            q[k + ps] = v.y;
        } else {
            q[k] = v;
        }
    };
    const S *M = static_cast<const S *>(j.moments);
    const R rho = ld(M, lc), ux = ld(M, n + lc), uy = ld(M, 2 * n + lc), uz = ld(M, 3 * n + lc);
    const R s4 = ld(M, 4 * n + lc), s5 = ld(M, 5 * n + lc), s6 = ld(M, 6 * n + lc), s7 = ld(M, 7 * n + lc),
            s8 = ld(M, 8 * n + lc);
    const R gx = lit<R>(adj_g<S>(d, 0)), gy = lit<R>(adj_g<S>(d, 1));
    R gz = lit<R>(adj_g<S>(d, 2));
    if (d.gz_field != nullptr) {
        const int64_t plane = (int64_t)d.nx * d.ny;
        const S *q = static_cast<const S *>(d.gz_field) + (plane * z + (int64_t)(ci.x & 0xFFFF) * d.nx + ((uint32_t)ci.x >> 16));
        if constexpr (TWO) gz = add_(gz, make_float2(q[0], q[plane]));
        else gz = add_(gz, q[0]);
    }
    const R om1 = lit<R>(S(1) - adj_omega<S>(d));
    const R half = lit<R>(S(0.5));

    // mu = S^T lambda_{t+1} (+ wall shear source)
    const S wss = adj_wss<S>(j);
    const S *ln = static_cast<const S *>(j.lam_next);
    R mu[Q];
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value, ib = opp_of(i), cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
        uint32_t pull = j.pull[ib];
        if constexpr (!TWO && cz == -1) pull += z == 0 ? (uint32_t)d.nz * ps : 0u;
        if constexpr (!TWO && cz == 1) pull -= z == d.nz - 1 ? (uint32_t)d.nz * ps : 0u;
        if constexpr (cx == 0 && cy == 0) {
            mu[i] = ld(ln, lc + (j.own[ib] + pull));
        } else {
            const uint32_t f = (uint32_t)((int32_t)(nb << (31 - nbit(cx, cy))) >> 31);
            const uint32_t dx = (cy == 0 ? 0u : (uint32_t)(cy < 0 ? ci.z : ci.w)) + (uint32_t)cx;
            mu[i] = ld(ln, (lc + (f & dx)) + j.own[ib] + (f & pull));
            if constexpr (OBJ == LBM_J_WSS && cz != 0)
                if (!f) mu[i] = add_(mu[i], lit<R>(wss * S(cz)));
        }
    });

    // q_k = sum_j mu_j C_kj (columns of (M^T)^{-1}), times 1 - omega
    const R e12 = add_(mu[1], mu[2]), e34 = add_(mu[3], mu[4]), e56 = add_(mu[5], mu[6]);
    const R q4 = mul_(lit<R>(S(0.25)), sub_(add_(mu[7], mu[10]), add_(mu[8], mu[9])));
    const R q5 = mul_(lit<R>(S(0.25)), sub_(add_(mu[11], mu[14]), add_(mu[12], mu[13])));
    const R q6 = mul_(lit<R>(S(0.25)), sub_(add_(mu[15], mu[18]), add_(mu[16], mu[17])));
    const R q7 = mul_(lit<R>(S(1.0 / 6.0)), fma_(lit<R>(-2), e34, add_(e12, e56)));
    const R q8 = mul_(lit<R>(S(1.0 / 6.0)), fma_(lit<R>(-2), e56, add_(e12, e34)));
    wterm = neg_(fma_(q4, s4, fma_(q5, s5, fma_(q6, s6, fma_(q7, s7, mul_(q8, s8))))));
    const R o4 = mul_(om1, q4), o5 = mul_(om1, q5), o6 = mul_(om1, q6), o7 = mul_(om1, q7), o8 = mul_(om1, q8);

    // contractions; Kabc: a, b, c derivatives along x, y, z
    const R ux3 = mul_(lit<R>(3), ux), uy3 = mul_(lit<R>(3), uy), uz3 = mul_(lit<R>(3), uz);
    const R uxh = mul_(half, ux), uyh = mul_(half, uy), uzh = mul_(half, uz);
    AxisSum<R> Y0[3], Y1[3];          // per c_x: over z (derivative 0, 1), then y
    R Y2[3];                          // second z derivative, plain in y
    sfor<0, 3>([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        AxisSum<R> T[3];
        sfor<0, 3>([&](auto bc) {
            constexpr int b = decltype(bc)::value;
            T[b] = axis_sum<R>(mu[dir_of(a - 1, b - 1, -1)], mu[dir_of(a - 1, b - 1, 0)], mu[dir_of(a - 1, b - 1, 1)], uz3, uzh, uz);
        });
        Y0[a] = axis_sum<R>(T[0].f0, T[1].f0, T[2].f0, uy3, uyh, uy);
        Y1[a] = axis_sum<R>(T[0].f1, T[1].f1, T[2].f1, uy3, uyh, uy);
        Y2[a] = axis_sum<R>(T[0].f2, T[1].f2, T[2].f2, uy3, uyh, uy).f0;
    });
    const AxisSum<R> X00 = axis_sum<R>(Y0[0].f0, Y0[1].f0, Y0[2].f0, ux3, uxh, ux);
    const AxisSum<R> X01 = axis_sum<R>(Y1[0].f0, Y1[1].f0, Y1[2].f0, ux3, uxh, ux);
    const AxisSum<R> X10 = axis_sum<R>(Y0[0].f1, Y0[1].f1, Y0[2].f1, ux3, uxh, ux);
    const R w0 = lit<R>(S(1.0 / 216.0)), w3 = lit<R>(S(1.0 / 72.0)), w9 = lit<R>(S(1.0 / 24.0));
    const R K000 = mul_(w0, X00.f0), K100 = mul_(w3, X00.f1), K200 = mul_(w3, X00.f2);
    const R K001 = mul_(w3, X01.f0), K101 = mul_(w9, X01.f1);
    const R K010 = mul_(w3, X10.f0), K110 = mul_(w9, X10.f1);
    const R K002 = mul_(w3, axis_sum<R>(Y2[0], Y2[1], Y2[2], ux3, uxh, ux).f0);
    const R K011 = mul_(w9, axis_sum<R>(Y1[0].f1, Y1[1].f1, Y1[2].f1, ux3, uxh, ux).f0);
    const R K020 = mul_(w3, axis_sum<R>(Y0[0].f2, Y0[1].f2, Y0[2].f2, ux3, uxh, ux).f0);

    // v = u - g / 2 (the bare velocity); the shear part of A_rho is -(v_a v_b - g_a g_b / 4), of
    // A_u minus 2 v or the other axis' v
    const R hx = mul_(half, gx), hy = mul_(half, gy), hz = mul_(half, gz);
    const R vx = sub_(ux, hx), vy = sub_(uy, hy), vz = sub_(uz, hz);
    const R xx = fma_(vx, vx, neg_(mul_(hx, hx))), yy = fma_(vy, vy, neg_(mul_(hy, hy))), zz = fma_(vz, vz, neg_(mul_(hz, hz)));
    R sh = mul_(o4, fma_(vx, vy, neg_(mul_(hx, hy))));
    sh = fma_(o5, fma_(vx, vz, neg_(mul_(hx, hz))), sh);
    sh = fma_(o6, fma_(vy, vz, neg_(mul_(hy, hz))), sh);
    sh = fma_(o7, sub_(xx, yy), sh);
    sh = fma_(o8, sub_(xx, zz), sh);
    const R Arho = sub_(fma_(hx, K100, fma_(hy, K010, fma_(hz, K001, K000))), sh);
    const R o78 = add_(o7, o8);
    // A_u / rho
    const R shx = fma_(o4, vy, fma_(o5, vz, mul_(mul_(lit<R>(2), o78), vx)));
    const R shy = fma_(o4, vx, fma_(o6, vz, mul_(mul_(lit<R>(-2), o7), vy)));
    const R shz = fma_(o5, vx, fma_(o6, vy, mul_(mul_(lit<R>(-2), o8), vz)));
    const R Bx = sub_(fma_(hx, K200, fma_(hy, K110, fma_(hz, K101, K100))), shx);
    const R By = sub_(fma_(hx, K110, fma_(hy, K020, fma_(hz, K011, K010))), shy);
    const R Az = sub_(fma_(hx, K101, fma_(hy, K011, fma_(hz, K002, K001))), shz);
    const R kap = lit<R>(adj_kappa<S>(j));
    const R Bz = OBJ == LBM_J_UBULK ? fma_(kap, recip_(rho), Az) : Az;
    const R base = sub_(Arho, fma_(Bx, vx, fma_(By, vy, mul_(Bz, vz))));

    // lambda_i = base + c_i . B + (1 - omega)(cx cy q4 + cx cz q5 + cy cz q6 + (cx^2 - cy^2) q7
    // + (cx^2 - cz^2) q8), split into one term per axis and the three cross terms; only the
    // terms with a non-zero lattice coefficient are added
    const R axm = sub_(o78, Bx), axp = add_(o78, Bx);     // cx = -1, +1
    const R aym = neg_(add_(o7, By)), ayp = sub_(By, o7);
    const R azm = neg_(add_(o8, Bz)), azp = sub_(Bz, o8);
    S *lo = static_cast<S *>(j.lam);
    // (the zero depends on the sums: no store address is formed before them)
    uint32_t bits;
    if constexpr (TWO) bits = __float_as_uint(K000.x);
    else bits = (uint32_t)__float_as_int((float)K000);
    const uint32_t wlc = lc + min(bits, j.zero);
    sfor<0, 9>([&](auto kc) {
        constexpr int k = decltype(kc)::value, cx = k % 3 - 1, cy = k / 3 - 1;
        R l = base;
        if constexpr (cx == 1) l = add_(l, axp);
        if constexpr (cx == -1) l = add_(l, axm);
        if constexpr (cy == 1) l = add_(l, ayp);
        if constexpr (cy == -1) l = add_(l, aym);
        if constexpr (cx * cy == 1) l = add_(l, o4);
        if constexpr (cx * cy == -1) l = sub_(l, o4);
        R t5 = azp, t6 = azm;                             // cz = +1, -1
        if constexpr (cx == 1) { t5 = add_(t5, o5); t6 = sub_(t6, o5); }
        if constexpr (cx == -1) { t5 = sub_(t5, o5); t6 = add_(t6, o5); }
        if constexpr (cy == 1) { t5 = add_(t5, o6); t6 = sub_(t6, o6); }
        if constexpr (cy == -1) { t5 = sub_(t5, o6); t6 = add_(t6, o6); }
        st(lo, j.own[dir_of(cx, cy, 0)] + wlc, l);
        st(lo, j.own[dir_of(cx, cy, 1)] + wlc, add_(l, t5));
        st(lo, j.own[dir_of(cx, cy, -1)] + wlc, add_(l, t6));
    });

    // accumulators: objective, dJ/dg_z, dJ/domega
    if constexpr (OBJ == LBM_J_UBULK) {
        jterm = mul_(kap, uz);
    } else {
        // the wall is a cylinder, so (cx, cy, +1) and (cx, cy, -1) are wall links together:
        // their terms are summed as the difference f*(+1) - f*(-1), formed from the
        // closed-form differences psi(+1) - psi(-1) = 6 u_z and psi'(+1) - psi'(-1) = 6
        // (the rest weights cancel exactly instead of in floating point)
        jterm = lit<R>(0);
        if (nb != 0x1FFu) {
            const R dZ0 = mul_(lit<R>(6), uz);
            auto psi = [](auto cc, R u, R &f, R &f1) {
                constexpr int c = decltype(cc)::value;
                if constexpr (c == 0) {
                    f = fma_(lit<R>(S(-1.5)), mul_(u, u), lit<R>(1));
                    f1 = mul_(lit<R>(-3), u);
                } else {
                    f = fma_(lit<R>(3), fma_(u, u, c > 0 ? u : neg_(u)), lit<R>(1));
                    f1 = fma_(lit<R>(6), u, lit<R>(3 * c));
                }
            };
            sfor<0, 9>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr int cx = k % 3 - 1, cy = k / 3 - 1;
                if constexpr (cx != 0 || cy != 0) {
                    constexpr int ip = dir_of(cx, cy, 1);
                    if (!((nb >> nbit(cx, cy)) & 1u)) {
                        R X0, X1, Yp, Yd;
                        psi(std::integral_constant<int, cx>{}, ux, X0, X1);
                        psi(std::integral_constant<int, cy>{}, uy, Yp, Yd);
                        const R x0y0 = mul_(X0, Yp);
                        const R dG = fma_(fma_(mul_(gx, X1), Yp, mul_(mul_(gy, X0), Yd)), dZ0, mul_(mul_(gz, x0y0), lit<R>(6)));
                        R t = mul_(mul_(lit<R>(S(w_of(ip))), rho), fma_(half, dG, mul_(x0y0, dZ0)));
                        if constexpr (cy == 0) t = fma_(om1, mul_(lit<R>(S(0.5 * cx)), s5), t);
                        if constexpr (cx == 0) t = fma_(om1, mul_(lit<R>(S(0.5 * cy)), s6), t);
                        jterm = fma_(lit<R>(wss), t, jterm);
                    }
                }
            });
        }
    }
    const R hrho = mul_(half, rho);
    R gterm = fma_(hrho, add_(K001, Az), mul_(hrho, fma_(o5, ux, fma_(o6, uy, mul_(mul_(lit<R>(-2), o8), uz)))));
    if constexpr (OBJ == LBM_J_UBULK) gterm = fma_(half, kap, gterm);
    S *seg = static_cast<S *>(j.acc_seg);
    st(seg, lc, add_(ld(seg, lc), gterm));
}

// End of a segment of the reverse sweep: its dJ/dg_z sums join the FP64 totals (dense cells).
template <class R>
__global__ void k_flush_segment(const Member *members, R *acc_seg, double *acc) {
    const Member &d = members[0];
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d.scells) return;
    const int z = (int)(s / d.Ps), r = (int)(s - (int64_t)z * d.Ps);
    const int4 ci = d.cellinfo[r];
    if (ci.x == -1) return;
    const int y = ci.x & 0xFFFF, x = (int)((uint32_t)ci.x >> 16);
    acc[((int64_t)z * d.ny + y) * d.nx + x] += (double)acc_seg[s];
    acc_seg[s] = R(0);
}

// FP32: planes 1 .. nz - 2 in pairs, ADJ_ZC / 2 pairs per thread, after the planes taken singly (as
// in k_odd2); FP64: every plane singly.  The objective and dJ/domega terms are summed per warp
// in a fixed order and added to the warp's own FP64 slots (deterministic), dJ/dg_z per cell.
template <int P, int OBJ>
__global__ void __launch_bounds__(ADJ_THREADS, P == LBM_F64 ? 3 : 4) k_adjoint(const __grid_constant__ AdjArgs j) {
    using S = typename Storage<P>::R;
    release_next_step();
    const AdjMember &d = j.one;
    const uint32_t zg = fastdiv(blockIdx.x, j.nb_mul, j.nb_shr);
    const uint32_t r = (blockIdx.x - zg * j.nb_plane) * ADJ_THREADS + threadIdx.x;
    const int4 ci = r < (uint32_t)d.Ps ? d.cellinfo[r] : make_int4(-1, 0, 0, 0);
    await_previous_step();
    S x0 = 0, x1 = 0;
    if (ci.x != -1) {
        const int singles = P == LBM_F64 ? d.nz : odd_single_planes(d.nz);
        if ((int)zg < singles) {
            const int z = P == LBM_F64 ? (int)zg : (zg == 0 ? 0 : d.nz - (int)zg);
            adjoint_cells<P, OBJ, S>(j, ci, r, z, x0, x1);
        } else if constexpr (P != LBM_F64) {
#pragma unroll 1
            for (int k = 0; k < ADJ_ZC / 2; ++k) {
                const int z = 1 + ((int)zg - singles) * ADJ_ZC + 2 * k;
                if (z + 2 >= d.nz) break;
                uint32_t rr = r;
                int4 cj = ci;
                asm volatile("" : "+r"(rr), "+r"(cj.x), "+r"(cj.y), "+r"(cj.z), "+r"(cj.w));    // nothing of a pass outlives it
                pf2 y0, y1;
                adjoint_cells<P, OBJ, pf2>(j, cj, rr, z, y0, y1);
                x0 += y0.x + y0.y;
                x1 += y1.x + y1.y;
            }
        }
    }
    // warp sums of the objective and omega terms in the compute type, added to the
    // warp's own FP64 slots (fixed order, no block barrier)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x0 += __shfl_down_sync(0xFFFFFFFFu, x0, o);
        x1 += __shfl_down_sync(0xFFFFFFFFu, x1, o);
    }
    if ((threadIdx.x & 31) == 0) {
        const int64_t wslot = (int64_t)blockIdx.x * (ADJ_THREADS / 32) + (threadIdx.x >> 5);
        j.blockacc[wslot] += (double)x0;
        j.blockacc[(int64_t)j.nblocks * (ADJ_THREADS / 32) + wslot] += (double)x1;
    }
}

// Column sums of up to five double arrays (stride n) into per-block partials.
static __global__ void __launch_bounds__(REDUCE_BLOCK) k_sum_columns(const double *base, int64_t n, int nv,
                                                                 double *partials) {
    __shared__ double sh[5 * 32];
    double acc[5] = {0, 0, 0, 0, 0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (k < nv) acc[k] += base[k * n + i];
    block_sum<5>(acc, sh);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 5; ++k) partials[blockIdx.x * 5 + k] = acc[k];
}

// ---- host launchers ------------------------------------------------------------------------------
#define LBM_DISPATCH_WP(WALL_, PAR_, ...)                                          \
    do {                                                                          \
        if (WALL_ == LBM_HALFWAY) {                                               \
            if (PAR_ == 0) { constexpr int W = LBM_HALFWAY, PA = 0; __VA_ARGS__; } \
            else { constexpr int W = LBM_HALFWAY, PA = 1; __VA_ARGS__; }          \
        } else if (WALL_ == LBM_FULLWAY) {                                        \
            if (PAR_ == 0) { constexpr int W = LBM_FULLWAY, PA = 0; __VA_ARGS__; } \
            else { constexpr int W = LBM_FULLWAY, PA = 1; __VA_ARGS__; }          \
        } else {                                                                  \
            if (PAR_ == 0) { constexpr int W = LBM_BOUZIDI, PA = 0; __VA_ARGS__; } \
            else { constexpr int W = LBM_BOUZIDI, PA = 1; __VA_ARGS__; }          \
        }                                                                         \
    } while (0)

static inline unsigned blocks_for(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

template <int P, int BS, int MINB, int ZC = 1>
cudaError_t launch_step_shape(int wall, int parity, bool stats, const StepArgs &a, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    LBM_DISPATCH_WP(wall, parity, {
        if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, BS, MINB, MODEL_MRT_H6, ZC>, a.nblocks_total, BS, a.overlap, a, s);
        else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, BS, MINB, MODEL_MRT_H6, ZC>, a.nblocks_total, BS, a.overlap, a, s);
    });
    return e;
}

template <int P, int BS, int MINB>
cudaError_t launch_step_pipe(int wall, int parity, bool stats, const StepArgs &a, cudaStream_t s) {
    using T = typename Storage<P>::T;
    const size_t smem = 2 * (size_t)Q * BS * sizeof(T);
    static int grid_cache[2][3][2] = {};            // resident blocks x SMs, per (parity, wall, stats)
    int &grid = grid_cache[parity][wall][stats ? 1 : 0];
    cudaError_t e = cudaSuccess;
    LBM_DISPATCH_WP(wall, parity, {
        auto kern = stats ? k_step_pipe<P, PA, W, EX_STATS, BS, MINB> : k_step_pipe<P, PA, W, EX_NONE, BS, MINB>;
        if (grid == 0) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            int per_sm = 0, dev = 0, sms = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, BS, smem);
            if (e == cudaSuccess) e = cudaGetDevice(&dev);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            grid = std::max(1, per_sm) * std::max(1, sms);
        }
        const int g = std::min(grid, a.nblocks_total);
        kern<<<g, BS, smem, s>>>(a);
    });
    return cudaGetLastError();
}

// The ablation models run in the thread count of shape 2.  The BGK and the second-order
// equilibrium fit its 64 registers on even and 72 on odd steps (128 before, when each
// population went through its own equilibrium); FP64, and general rates, which hold 27
// populations and 23 moments, take half the resident blocks.
template <int P, int BS, int MINB>
cudaError_t launch_step_model(int wall, int parity, bool stats, const StepArgs &a, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    constexpr int MINB_R = MINB > 1 ? MINB / 2 : 1;
    LBM_DISPATCH_WP(wall, parity, {
        constexpr int MINB_C = P == LBM_F64 ? MINB_R : MINB - PA;
        switch (a.collision) {
            case MODEL_BGK:
                if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, BS, MINB_C, MODEL_BGK>, a.nblocks_total, BS, a.overlap, a, s);
                else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, BS, MINB_C, MODEL_BGK>, a.nblocks_total, BS, a.overlap, a, s);
                break;
            case MODEL_O2:
                if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, BS, MINB_C, MODEL_O2>, a.nblocks_total, BS, a.overlap, a, s);
                else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, BS, MINB_C, MODEL_O2>, a.nblocks_total, BS, a.overlap, a, s);
                break;
            case MODEL_BGK | MODEL_O2:
                if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, BS, MINB_C, MODEL_BGK | MODEL_O2>, a.nblocks_total, BS, a.overlap, a, s);
                else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, BS, MINB_C, MODEL_BGK | MODEL_O2>, a.nblocks_total, BS, a.overlap, a, s);
                break;
            case MODEL_RATES:
                if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, BS, MINB_R, MODEL_RATES>, a.nblocks_total, BS, a.overlap, a, s);
                else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, BS, MINB_R, MODEL_RATES>, a.nblocks_total, BS, a.overlap, a, s);
                break;
            case MODEL_RATES | MODEL_O2:
                if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, BS, MINB_R, MODEL_RATES | MODEL_O2>, a.nblocks_total, BS, a.overlap, a, s);
                else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, BS, MINB_R, MODEL_RATES | MODEL_O2>, a.nblocks_total, BS, a.overlap, a, s);
                break;
            default: return cudaErrorInvalidValue;
        }
    });
    return e;
}

// A step of a compact pipe context on pairs of cells, in shape V.
template <int P, int V, int WALL, class A>
cudaError_t launch_pair_args(int parity, bool stats, int blocks, bool overlap, const A &a, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    constexpr StepShape S = STEP_SHAPES[V];
    if (parity == 0) {
        if (stats) e = launch_step_kernel<A>(k_even2<P, WALL, EX_STATS, EVEN2_THREADS, EVEN2_BLOCKS<P, WALL>, A>, blocks, EVEN2_THREADS, overlap, a, s);
        else e = launch_step_kernel<A>(k_even2<P, WALL, EX_NONE, EVEN2_THREADS, EVEN2_BLOCKS<P, WALL>, A>, blocks, EVEN2_THREADS, overlap, a, s);
    } else {
        if (stats) e = launch_step_kernel<A>(k_odd2<P, WALL, EX_STATS, S.pt, S.pb, S.pz, A>, blocks, S.pt, overlap, a, s);
        else e = launch_step_kernel<A>(k_odd2<P, WALL, EX_NONE, S.pt, S.pb, S.pz, A>, blocks, S.pt, overlap, a, s);
    }
    return e;
}

// (the lattice functions folded by the compiler: evaluated per launch they took 4 us)
template <class A, int... I>
void fill_pull(A &o, uint32_t stride, uint32_t ps, std::integer_sequence<int, I...>) {
    constexpr int jump[] = {(opp_of(I) - I)...}, cz[] = {cz_of(I)...};
    for (int i = 0; i < Q; ++i) {
        o.own[i] = (uint32_t)i * stride;
        o.pull[i] = (uint32_t)jump[i] * stride - (uint32_t)cz[i] * ps;
    }
}

template <int V>
void fill_pair_one(PairArgsOne &o, const StepArgs &a, const Member *hm) {
    fill_pair_args(o, a);
    fill_pair_member(o.one, hm[0]);
    o.stf[0] = a.stf[0];
    o.nb_plane = (uint32_t)((hm[0].Ps + STEP_SHAPES[V].pt - 1) / STEP_SHAPES[V].pt);
    fastdiv_setup(o.nb_plane, o.nb_mul, o.nb_shr);
    fill_pull(o, (uint32_t)a.stride, (uint32_t)hm[0].Ps, std::make_integer_sequence<int, Q>{});
}

template <int P, int V>
cudaError_t launch_pair(int wall, int parity, bool stats, const StepArgs &a, const Member *hm, cudaStream_t s) {
    if (a.n_members == 1) {
        PairArgsOne o;
        fill_pair_one<V>(o, a, hm);
        return wall == LBM_BOUZIDI ? launch_pair_args<P, V, LBM_BOUZIDI>(parity, stats, a.nblocks_total, a.overlap, o, s)
                                   : launch_pair_args<P, V, LBM_HALFWAY>(parity, stats, a.nblocks_total, a.overlap, o, s);
    }
    PairArgsMany o;
    fill_pair_args(o, a);
    o.n_members = a.n_members;
    fill_pull(o, (uint32_t)a.stride, 0u, std::make_integer_sequence<int, Q>{});
    for (int m = 0; m < a.n_members; ++m) {
        o.stf[m] = a.stf[m];
        fill_pair_member(o.many[m], hm[m]);
        o.nb_plane[m] = (uint32_t)((hm[m].Ps + STEP_SHAPES[V].pt - 1) / STEP_SHAPES[V].pt);
        fastdiv_setup(o.nb_plane[m], o.nb_mul[m], o.nb_shr[m]);
    }
    for (int m = 0; m <= a.n_members; ++m) o.block0[m] = a.block0[m];
    return wall == LBM_BOUZIDI ? launch_pair_args<P, V, LBM_BOUZIDI>(parity, stats, a.nblocks_total, a.overlap, o, s)
                               : launch_pair_args<P, V, LBM_HALFWAY>(parity, stats, a.nblocks_total, a.overlap, o, s);
}

// A shape of several planes per thread: pairs of cells in the compact pipe layouts, else the
// planes one after the other, or one plane per thread (make_args decides).
template <int P, int V>
cudaError_t launch_planes(int wall, int parity, bool stats, const StepArgs &a, const Member *hm, cudaStream_t s) {
    if (a.pairs) return launch_pair<P, V>(wall, parity, stats, a, hm, s);
    constexpr StepShape S = STEP_SHAPES[V];
    if (a.single) return launch_step_shape<P, SINGLE_THREADS, STEP_SHAPES[SINGLE_VARIANT].min_blocks>(wall, parity, stats, a, s);
    const bool full = wall == LBM_FULLWAY;
    cudaError_t e = cudaSuccess;
    auto go = [&](auto pa, auto w) {
        constexpr int PA = decltype(pa)::value, W = decltype(w)::value;
        if (stats) e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_STATS, S.threads, S.min_blocks, MODEL_MRT_H6, S.zc>, a.nblocks_total, S.threads, a.overlap, a, s);
        else e = launch_step_kernel<StepArgs>(k_step<P, PA, W, EX_NONE, S.threads, S.min_blocks, MODEL_MRT_H6, S.zc>, a.nblocks_total, S.threads, a.overlap, a, s);
    };
    using std::integral_constant;
    if (full && parity == 0) go(integral_constant<int, 0>{}, integral_constant<int, LBM_FULLWAY>{});
    else if (full) go(integral_constant<int, 1>{}, integral_constant<int, LBM_FULLWAY>{});
    else if (parity == 0) go(integral_constant<int, 0>{}, integral_constant<int, LBM_HALFWAY>{});
    else go(integral_constant<int, 1>{}, integral_constant<int, LBM_HALFWAY>{});
    return e;
}

template <int P>
cudaError_t launch_step(int wall, int parity, bool stats, const StepArgs &a, const Member *hm, int variant,
                        cudaStream_t s) {
    if (a.nblocks_total <= 0) return cudaSuccess;
    if (a.collision == MODEL_MRT_H6 && STEP_SHAPES[variant].staged)
        return launch_step_staged<P>(wall, parity, stats, a, variant, s);
    if (a.collision != MODEL_MRT_H6) {
        if constexpr (P == LBM_F64) return launch_step_model<P, STEP_SHAPE_F64.threads, STEP_SHAPE_F64.min_blocks>(wall, parity, stats, a, s);
        else if constexpr (P == LBM_F32) return launch_step_model<P, 128, 8>(wall, parity, stats, a, s);
        else return cudaErrorInvalidValue;
    }
    if constexpr (P == LBM_F64) {
        return launch_step_shape<P, STEP_SHAPE_F64.threads, STEP_SHAPE_F64.min_blocks>(wall, parity, stats, a, s);
    } else {
        switch (variant) {
            case 1: return launch_step_shape<P, 256, 3>(wall, parity, stats, a, s);
            case 2: return launch_step_shape<P, 128, 8>(wall, parity, stats, a, s);
            case 3: return launch_step_shape<P, 512, 2>(wall, parity, stats, a, s);
            case 4:
                if constexpr (P == LBM_F32) return launch_step_pipe<P, 256, 3>(wall, parity, stats, a, s);
                else return cudaErrorInvalidValue;
            case 5:
                if constexpr (P == LBM_F32) return launch_step_pipe<P, 128, 6>(wall, parity, stats, a, s);
                else return cudaErrorInvalidValue;
            case 6: return launch_planes<P, 6>(wall, parity, stats, a, hm, s);
            case 7: return launch_planes<P, 7>(wall, parity, stats, a, hm, s);
            case 8: return launch_planes<P, 8>(wall, parity, stats, a, hm, s);
            case 9: return launch_planes<P, 9>(wall, parity, stats, a, hm, s);
            case 10: return launch_planes<P, 10>(wall, parity, stats, a, hm, s);
            default: return launch_step_shape<P, 256, 4>(wall, parity, stats, a, s);
        }
    }
}

// Forward step of a single half-way pipe that also stores the adjoint moments (F32, F64).
template <int P>
cudaError_t launch_step_moments(int parity, const StepArgs &a, const Member *hm, cudaStream_t s) {
    if constexpr (P == LBM_F32) {
        if (a.pairs) {
            PairArgsOne o;
            constexpr StepShape S = STEP_SHAPES[MOM_VARIANT_PAIRS];
            fill_pair_one<MOM_VARIANT_PAIRS>(o, a, hm);
            if (parity == 0)
                return launch_step_kernel<PairArgsOne>(k_even2<P, LBM_HALFWAY, EX_MOMENTS, EVEN2_THREADS, EVEN2_BLOCKS<P, LBM_HALFWAY>, PairArgsOne>, a.nblocks_total, EVEN2_THREADS, a.overlap, o, s);
            return launch_step_kernel<PairArgsOne>(k_odd2<P, LBM_HALFWAY, EX_MOMENTS, S.pt, S.pb, S.pz, PairArgsOne>, a.nblocks_total, S.pt, a.overlap, o, s);
        }
    }
    if constexpr (P == LBM_F64 || P == LBM_F32) {
        constexpr int BS = P == LBM_F64 ? STEP_SHAPE_F64.threads : 256, MINB = P == LBM_F64 ? STEP_SHAPE_F64.min_blocks : 4;
        constexpr int ZC = 1;
        if (parity == 0)
            return launch_step_kernel<StepArgs>(k_step<P, 0, LBM_HALFWAY, EX_MOMENTS, BS, MINB, MODEL_MRT_H6, ZC>, a.nblocks_total, BS, a.overlap, a, s);
        return launch_step_kernel<StepArgs>(k_step<P, 1, LBM_HALFWAY, EX_MOMENTS, BS, MINB, MODEL_MRT_H6, ZC>, a.nblocks_total, BS, a.overlap, a, s);
    } else {
        return cudaErrorNotSupported;
    }
}

template <int P>
cudaError_t launch_sum_columns(const double *base, int64_t n, int nv, double *partials, int n_partials_max,
                               double *out, cudaStream_t s) {
    int nb = (int)blocks_for(n, REDUCE_BLOCK);
    if (nb > n_partials_max) nb = n_partials_max;
    if (nb < 1) nb = 1;
    k_sum_columns<<<nb, REDUCE_BLOCK, 0, s>>>(base, n, nv, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_final<<<1, REDUCE_BLOCK, 0, s>>>(partials, nb, out);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_adjoint(bool overlap, const AdjArgs &j, cudaStream_t s) {
    if constexpr (P == LBM_F64 || P == LBM_F32) {
        if (j.objective == LBM_J_UBULK) return launch_step_kernel<AdjArgs>(k_adjoint<P, LBM_J_UBULK>, j.nblocks, ADJ_THREADS, overlap, j, s);
        return launch_step_kernel<AdjArgs>(k_adjoint<P, LBM_J_WSS>, j.nblocks, ADJ_THREADS, overlap, j, s);
    } else {
        return cudaErrorNotSupported;
    }
}

// Everything about the pipe and the launch that stays the same over the sweep.
template <int... I>
void fill_adjoint_index(AdjArgs &j, std::integer_sequence<int, I...>) {
    constexpr int jump[] = {(opp_of(I) - I)...}, cz[] = {cz_of(I)...};
    for (int i = 0; i < Q; ++i) {
        j.own[i] = (uint32_t)i * j.one.n;
        j.pull[i] = (uint32_t)jump[i] * j.one.n - (uint32_t)cz[i] * (uint32_t)j.one.Ps;
    }
}
template <int P>
void prepare_adjoint(AdjArgs &j, const Member &d) {
    AdjMember &o = j.one;
    o.cellinfo = d.cellinfo;
    o.gz_field = d.gz_field;
    o.nx = d.nx; o.ny = d.ny; o.nz = d.nz; o.Ps = d.Ps;
    o.n = (uint32_t)d.scells;
    for (int k = 0; k < 3; ++k) {
        o.g[k] = d.g[k];
        o.gf[k] = d.gf[k];
    }
    o.omega = d.omega;
    o.omegaf = d.omegaf;
    j.zero = 0;
    j.nb_plane = (uint32_t)((d.Ps + ADJ_THREADS - 1) / ADJ_THREADS);
    fastdiv_setup(j.nb_plane, j.nb_mul, j.nb_shr);
    j.nblocks = (int32_t)(j.nb_plane * (P == LBM_F64 ? d.nz : odd_single_planes(d.nz) + odd_pair_groups(d.nz, ADJ_ZC)));
    fill_adjoint_index(j, std::make_integer_sequence<int, Q>{});
}

template <int P>
cudaError_t launch_flush_segment(const StepArgs &a, const Member &hm, const AdjArgs &j, cudaStream_t s) {
    using R = typename Storage<P>::R;
    if constexpr (P == LBM_F64 || P == LBM_F32) {
        k_flush_segment<R><<<blocks_for(hm.scells, 256), 256, 0, s>>>(a.members, static_cast<R *>(j.acc_seg), j.acc);
        return cudaGetLastError();
    } else {
        return cudaErrorNotSupported;
    }
}

template <int P>
cudaError_t launch_moments(int wall, int parity, const StepArgs &a, const Member &hm, int m, void *rho,
                           void *u, cudaStream_t s) {
    using R = typename Storage<P>::R;
    if (hm.cells == 0) return cudaSuccess;
    LBM_DISPATCH_WP(wall, parity, {
        k_moments<P, PA, W><<<blocks_for(hm.cells, 256), 256, 0, s>>>(a, m, (R *)rho, (R *)u);
    });
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_get_pops(int wall, int parity, const StepArgs &a, const Member &hm, int m, double *f,
                            cudaStream_t s) {
    if (hm.cells == 0) return cudaSuccess;
    LBM_DISPATCH_WP(wall, parity, { k_get_pops<P, PA, W><<<blocks_for(hm.cells, 256), 256, 0, s>>>(a, m, f); });
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_set_pops(int wall, int parity, const StepArgs &a, const Member &hm, int m, const double *f,
                            cudaStream_t s) {
    if (hm.cells == 0) return cudaSuccess;
    LBM_DISPATCH_WP(wall, parity, { k_set_pops<P, PA, W><<<blocks_for(hm.cells, 256), 256, 0, s>>>(a, m, f); });
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_init(int wall, const StepArgs &a, const Member &hm, int m, int profile, double noise_amp,
                        uint64_t seed, const double *rho, const double *u, cudaStream_t s) {
    if (hm.cells == 0) return cudaSuccess;
    const unsigned nb = blocks_for(hm.cells, 256);
    if (wall == LBM_HALFWAY) k_init<P, LBM_HALFWAY><<<nb, 256, 0, s>>>(a, m, profile, noise_amp, seed, rho, u);
    else if (wall == LBM_FULLWAY) k_init<P, LBM_FULLWAY><<<nb, 256, 0, s>>>(a, m, profile, noise_amp, seed, rho, u);
    else k_init<P, LBM_BOUZIDI><<<nb, 256, 0, s>>>(a, m, profile, noise_amp, seed, rho, u);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_reduce(int wall, int parity, const StepArgs &a, const Member &hm, int m, double *partials,
                          int n_partials_max, double *out, cudaStream_t s) {
    int nb = (int)blocks_for(hm.cells, REDUCE_BLOCK);
    if (nb > n_partials_max) nb = n_partials_max;
    if (nb < 1) nb = 1;
    LBM_DISPATCH_WP(wall, parity, { k_reduce<P, PA, W><<<nb, REDUCE_BLOCK, 0, s>>>(a, m, partials); });
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_final<<<1, REDUCE_BLOCK, 0, s>>>(partials, nb, out);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_force_tables(const Member *dmembers, const Member &hm, int m, void *ftab, void *ztab,
                                cudaStream_t s) {
    using R = typename Storage<P>::R;
    const int n = (int)std::max<int64_t>((int64_t)hm.nx * hm.ny, hm.nz);
    k_force_tables<R><<<blocks_for(n, 256), 256, 0, s>>>(dmembers, m, (R *)ftab, (R *)ztab);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_modes(int wall, int parity, const StepArgs &a, const Member &hm, int m, const ModesArgs &ma,
                         double *E, cudaStream_t s) {
    (void)hm;
    const int nblk = ma.n_sections * ma.n_rings;
    const size_t shm = 3 * (size_t)ma.n_theta * sizeof(double);
    LBM_DISPATCH_WP(wall, parity, {
        if (shm > 48 * 1024) {
            // the limit is the kernel's, which every context and thread shares: always the largest
            // ring's, so that no call lowers it between another's limit and launch
            cudaError_t e = cudaFuncSetAttribute(k_modes<P, PA, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 3 * MODES_MAX_THETA * (int)sizeof(double));
            if (e != cudaSuccess) return e;
        }
        k_modes<P, PA, W><<<nblk, MODES_BLOCK, shm, s>>>(a, m, ma, E);
    });
    return cudaGetLastError();
}

}  // namespace lbm

// Explicit instantiation of every launcher for one storage precision.
#define LBM_INSTANTIATE(P)                                                                              \
    namespace lbm {                                                                                     \
    template cudaError_t launch_step<P>(int, int, bool, const StepArgs &, const Member *, int,            \
                                         cudaStream_t);                                                  \
    template cudaError_t launch_step_moments<P>(int, const StepArgs &, const Member *, cudaStream_t);     \
    template cudaError_t launch_adjoint<P>(bool, const AdjArgs &, cudaStream_t);                         \
    template void prepare_adjoint<P>(AdjArgs &, const Member &);                                         \
    template cudaError_t launch_flush_segment<P>(const StepArgs &, const Member &, const AdjArgs &,       \
                                                 cudaStream_t);                                          \
    template cudaError_t launch_sum_columns<P>(const double *, int64_t, int, double *, int, double *,    \
                                               cudaStream_t);                                            \
    template cudaError_t launch_moments<P>(int, int, const StepArgs &, const Member &, int, void *,     \
                                           void *, cudaStream_t);                                       \
    template cudaError_t launch_get_pops<P>(int, int, const StepArgs &, const Member &, int, double *,  \
                                            cudaStream_t);                                              \
    template cudaError_t launch_set_pops<P>(int, int, const StepArgs &, const Member &, int,            \
                                            const double *, cudaStream_t);                              \
    template cudaError_t launch_init<P>(int, const StepArgs &, const Member &, int, int, double,        \
                                        uint64_t, const double *, const double *, cudaStream_t);        \
    template cudaError_t launch_reduce<P>(int, int, const StepArgs &, const Member &, int, double *,    \
                                          int, double *, cudaStream_t);                                 \
    template cudaError_t launch_modes<P>(int, int, const StepArgs &, const Member &, int,               \
                                         const ModesArgs &, double *, cudaStream_t);                    \
    template cudaError_t launch_force_tables<P>(const Member *, const Member &, int, void *, void *,     \
                                                cudaStream_t);                                          \
    }

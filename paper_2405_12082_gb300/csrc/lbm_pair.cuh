// lbm_pair.cuh -- the step of the compact pipe layouts with two cells per thread on the
// paired FP32 instructions (F32, F16S and BF16 storage, half-way and Bouzidi walls).
//
// Even steps (k_even2): own slots only, so a thread takes two cells that are neighbours in x
// (an even storage position and the next one: rows start on 64-byte boundaries) and moves
// each population of the pair with one access of twice the width.  No neighbour data is
// needed: the 27 loads do not wait for the position table.
// Odd steps (k_odd2): neighbour slots, which an x pair could only reach with misaligned
// accesses, so a thread takes the planes z and z + 1 of one position: the same table entry,
// row offsets, wall links (the wall is a cylinder), link coefficients and, one plane apart,
// addresses serve both cells, and a warp's accesses stay contiguous.
//
// Why pairs: the step is bound by DRAM (F32) or by the instructions issued per cell at the
// warps that fit an SM (16-bit).  FFMA2 halves the arithmetic's issue slots (285 -> 145 per
// cell, F32 330 -> 165) and the pair shares the rest: F16S on the R = 48 pipe 703 -> 359 (even)
// and 885 -> 542 (odd) warp instructions per 32 cells, at the same number of cells per SM (14-20
// warps of 64 or 128 cells against 32 of 32).  Measured on the R = 96 pipe, one cell per thread
// against pairs (us per even / odd step, timed apart): F32 1143 / 1267 -> 1066 / 1166, F16S
// 913 / 1040 -> 639 / 861, BF16 908 / 1088 -> 630 / 867.
#pragma once

#include "lbm_internal.h"

namespace lbm {

// ---- storage of a pair ------------------------------------------------------------------
// Values stay in storage units (the scaled half format is collided scaled).
template <int P> struct PairStorage;
template <> struct PairStorage<LBM_F32> {
    using T = float; using V = float2;
    static __device__ __forceinline__ pf2 up(V v) { return v; }
    static __device__ __forceinline__ V down(pf2 v) { return v; }
    using B = float;                     // how a scalar access carries it
    static __device__ __forceinline__ float up1(B v) { return v; }
    static __device__ __forceinline__ B down1(float v) { return v; }
};
template <> struct PairStorage<LBM_F16S> {
    using T = __half; using V = __half2;
    static __device__ __forceinline__ pf2 up(V v) { return __half22float2(v); }
    static __device__ __forceinline__ V down(pf2 v) { return __float22half2_rn(v); }
    using B = uint16_t;
    static __device__ __forceinline__ float up1(B v) { return __half2float(__ushort_as_half(v)); }
    static __device__ __forceinline__ B down1(float v) { return __half_as_ushort(__float2half_rn(v)); }
};
template <> struct PairStorage<LBM_BF16> {
    using T = __nv_bfloat16; using V = __nv_bfloat162;
    static __device__ __forceinline__ pf2 up(V v) { return __bfloat1622float2(v); }
    static __device__ __forceinline__ V down(pf2 v) { return __float22bfloat162_rn(v); }
    using B = uint16_t;
    static __device__ __forceinline__ float up1(B v) { return __bfloat162float(__ushort_as_bfloat16(v)); }
    static __device__ __forceinline__ B down1(float v) { return __bfloat16_as_ushort(__float2bfloat16_rn(v)); }
};

// ---- what a block works on --------------------------------------------------------------
// Members travel in the kernel parameters (their fields are then constants of the launch, not
// loads); an ensemble looks its member up by block.
struct PairTask {
    uint32_t local;      // block index inside the member
    int m;
};
template <class A>
__device__ __forceinline__ PairTask pair_task(const A &a) {
    if constexpr (A::kOne) {
        return PairTask{blockIdx.x, 0};
    } else {
        int lo = 0, hi = a.n_members - 1;
        while (lo < hi) {          // largest m with block0[m] <= blk
            const int mid = (lo + hi + 1) >> 1;
            if (a.block0[mid] <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        return PairTask{(uint32_t)((int)blockIdx.x - a.block0[lo]), lo};
    }
}
template <class A>
__device__ __forceinline__ const auto &pair_member(const A &a, int m) {
    if constexpr (A::kOne) return a.one;
    else return a.many[m];
}
template <class A>
__device__ __forceinline__ float pair_st(const A &a, int m) {
    return a.times ? a.times[a.tidx].stf[m] : a.stf[m];
}
template <class A>
__device__ __forceinline__ int64_t pair_t(const A &a) { return a.times ? a.times[a.tidx].t : a.t; }

// ---- even step ----------------------------------------------------------------------------
// The default model on the cells of a pair kernel: F32 in its pinned order, the 16-bit formats in
// the shorter form.
template <int P, bool ACT, class R, class Emit>
__device__ __forceinline__ Macro<R> pair_collide(const MomentSums<R> &ms, R gx, R gy, R gz, float omega, float inv, float sc,
                                                 R *s_out, Emit &&emit, R act = lit<R>(1)) {
    if constexpr (P == LBM_F32) return collide_f32<R, ACT>(ms, gx, gy, gz, omega, s_out, emit, act);
    else return collide_mrt<R, P == LBM_F16S, ACT, true>(ms, gx, gy, gz, omega, inv, sc, s_out, emit, act);
}

// The pair at stored positions lc, lc + 1 (plane z, position r, table entry pi with its first
// cell fluid), whose populations are in raw.
template <int P, int WALL, int EXTRA, class A, class D>
__device__ __forceinline__ void even_pair(const A &a, const D &d, int m, uint32_t lc, uint32_t z, uint32_t r, uint32_t pi,
                                          const typename PairStorage<P>::V (&raw)[Q]) {
    using PS = PairStorage<P>;
    using T = typename PS::T;
    using V = typename PS::V;
    char *const base = static_cast<char *>(a.pops);
    const uint64_t stb = (uint64_t)a.stride * sizeof(T);
    const uint32_t vo = ((uint32_t)d.off + lc) * (uint32_t)sizeof(T);
    const uint32_t col = pi >> PAIR_SHIFT;
    const pf2 act = make_float2(1.f, (pi & PAIR_B) ? 1.f : 0.f);
    // acceleration (see acceleration())
    pf2 gx = lit<pf2>(d.gf[0]), gy = lit<pf2>(d.gf[1]), gz = lit<pf2>(d.gf[2]);
    const int64_t plane = (int64_t)d.nx * d.ny;
    if (d.gz_field != nullptr) {
        const float *q = static_cast<const float *>(d.gz_field) + (plane * z + col);
        gz.x += q[0];
        if (pi & PAIR_B) gz.y += q[1];
    }
    if (d.trig && pair_t(a) < d.t_end) {
        const float st = pair_st(a, m);
        const float *zt = static_cast<const float *>(d.ztab);
        const float2 *ft = reinterpret_cast<const float2 *>(d.ftabc) + (r >> 1);
        const pf2 sc = lit<pf2>(st * zt[z]), ss = lit<pf2>(st * zt[d.nz + z]);
        const uint32_t hp = (uint32_t)d.Ps >> 1;
        gx = fma_(sc, ft[0], gx);
        gy = fma_(sc, ft[hp], gy);
        gz = fma_(ss, ft[2 * hp], gz);
    }
    pf2 v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = PS::up(raw[i]);
    if constexpr (WALL == LBM_BOUZIDI) {
        if (pi & PAIR_WALL) {
            const float *tab = static_cast<const float *>(d.dtab) + (int64_t)col * 27;
            sfor<0, Q>([&](auto jc) {
                constexpr int j = decltype(jc)::value, cx = cx_of(j), cy = cy_of(j);
                if constexpr (cx != 0 || cy != 0) {        // C is zero for links that meet no wall
                    const pf2 C = make_float2(tab[nbit(cx, cy) * 3 + 2], (pi & PAIR_B) ? tab[27 + nbit(cx, cy) * 3 + 2] : 0.f);
                    v[opp_of(j)] = make_float2(C.x != 0.f ? fma_(C.x, v[j].x, v[opp_of(j)].x) : v[opp_of(j)].x,
                                               C.y != 0.f ? fma_(C.y, v[j].y, v[opp_of(j)].y) : v[opp_of(j)].y);
                }
            });
        }
    }
    const MomentSums<pf2> ms = moment_sums<pf2, P == LBM_F32>(v);
    Macro<pf2> mm;
    // a slot is written where it was read: the zero keeps the compiler from carrying the 27
    // addresses through the collision in registers
    char *const wbase = base + a.zero;
    const uint32_t wo = vo + a.zero;
    auto store = [&](auto ic, pf2 f) {
        constexpr int ib = opp_of(decltype(ic)::value);
        *reinterpret_cast<V *>(wbase + ib * stb + wo) = PS::down(f);
    };
    if constexpr (WALL == LBM_BOUZIDI) {
        mm = pair_collide<P, true, pf2>(ms, gx, gy, gz, d.omegaf, a.f16_inv, a.f16_scale, nullptr,
                                        [&](auto ic, pf2 f) { v[decltype(ic)::value] = f; }, act);
        if (pi & PAIR_WALL) {
            const float *tab = static_cast<const float *>(d.dtab) + (int64_t)col * 27;
            const uint32_t nbA = (uint32_t)d.cellinfo[r].y, nbB = (uint32_t)d.cellinfo[r + 1].y;
            sfor<0, Q>([&](auto jc) {
                constexpr int j = decltype(jc)::value, cx = cx_of(j), cy = cy_of(j), k = nbit(cx, cy);
                if constexpr (cx != 0 || cy != 0) {
                    pf2 f = v[j];
                    const pf2 o = v[opp_of(j)];
                    if (!((nbA >> k) & 1u)) f.x = fma_(tab[k * 3], f.x, mul_(tab[k * 3 + 1], o.x));
                    if ((pi & PAIR_B) && !((nbB >> k) & 1u)) f.y = fma_(tab[27 + k * 3], f.y, mul_(tab[27 + k * 3 + 1], o.y));
                    store(jc, f);
                } else {
                    store(jc, v[j]);
                }
            });
        } else {
            sfor<0, Q>([&](auto jc) { store(jc, v[decltype(jc)::value]); });
        }
    } else {
        pf2 sk[5];
        mm = pair_collide<P, true, pf2>(ms, gx, gy, gz, d.omegaf, a.f16_inv, a.f16_scale,
                                        EXTRA == EX_MOMENTS ? sk : nullptr, store, act);
        if constexpr (EXTRA == EX_MOMENTS) {
            pf2 *mo = reinterpret_cast<pf2 *>(static_cast<float *>(a.moments) + lc);
            const int64_t n = d.scells >> 1;
            mo[0] = mm.rho;
            mo[n] = mm.ux;
            mo[2 * n] = mm.uy;
            mo[3 * n] = mm.uz;
#pragma unroll
            for (int k = 0; k < 5; ++k) mo[(4 + k) * n] = sk[k];
        }
    }
    if constexpr (EXTRA == EX_STATS) {
        const int64_t cell = d.doff + plane * z + col;
        add_stats(a.stats + cell, a.dstride, (double)mm.uz.x);
        if (pi & PAIR_B) add_stats(a.stats + cell + 1, a.dstride, (double)mm.uz.y);
    }
}

// Two pairs per thread in the 16-bit formats with half-way walls (even_pairs): one 8-byte access
// loads a population of four cells, so the second pair's values wait in 27 registers while the
// first is collided, and the addresses serve both (R = 96 pipe, when it was made: BF16 750 -> 662
// us, F16S 687 -> 681; now 630 and 639).  In F32 the second pair would take 54 registers, and with Bouzidi walls the outputs of a
// pair are held as well (860 -> 1,002 us in F16S): one pair there.
template <int P, int WALL, int EXTRA, int BS, int MINB, class A>
__global__ void __launch_bounds__(BS, MINB) k_even2(const __grid_constant__ A a) {
    using PS = PairStorage<P>;
    using T = typename PS::T;
    using V = typename PS::V;
    constexpr int NP = even_pairs(P, WALL);
    release_next_step();
    const PairTask tk = pair_task(a);
    const auto &d = pair_member(a, tk.m);
    const uint32_t group = tk.local * BS + threadIdx.x;
    if (group >= (uint32_t)(d.scells / (2 * NP))) return;
    const uint32_t lc = 2 * NP * group;
    const char *const base = static_cast<const char *>(a.pops);
    const uint64_t stb = (uint64_t)a.stride * sizeof(T);
    const uint32_t vo = ((uint32_t)d.off + lc) * (uint32_t)sizeof(T);
    const uint32_t z = fastdiv(lc, d.ps_mul, d.ps_shr);
    const uint32_t r = lc - z * (uint32_t)d.Ps;
    if constexpr (NP == 1) {
        const uint32_t pi = d.pairinfo[r >> 1];
        await_previous_step();
        V raw[Q];
        sfor<0, Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            raw[i] = *reinterpret_cast<const V *>(base + i * stb + vo);
        });
        if (pi & PAIR_A) even_pair<P, WALL, EXTRA>(a, d, tk.m, lc, z, r, pi, raw);
    } else {
        const uint2 pi = *reinterpret_cast<const uint2 *>(d.pairinfo + (r >> 1));
        await_previous_step();
        V first[Q], second[Q];
        sfor<0, Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            const uint2 w = *reinterpret_cast<const uint2 *>(base + i * stb + vo);
            first[i] = *reinterpret_cast<const V *>(&w.x);
            second[i] = *reinterpret_cast<const V *>(&w.y);
        });
        // (a row's cells come before its padding: without a cell in the first pair the second has none)
        if (!(pi.x & PAIR_A)) return;
        even_pair<P, WALL, EXTRA>(a, d, tk.m, lc, z, r, pi.x, first);
        if (pi.y & PAIR_A) even_pair<P, WALL, EXTRA>(a, d, tk.m, lc + 2, z, r + 2, pi.y, second);
    }
}

// ---- odd step -----------------------------------------------------------------------------
// Direction i is read at element (relative to the position's own element of plane zA in array
// 0): f ? ib st - cz Ps + (row offset of y - cy) - cx : i st, f the fluid bit of x - c_i;
// f*_i is written where direction ib is read.  As own + (f-mask & difference): the own part
// and the difference are constants of the context (kOne: kernel parameters).
template <int I, class A, class D>
__device__ __forceinline__ uint32_t own_at(const A &a, const D &d) {
    return a.own[I];
}
template <int I, class A, class D>
__device__ __forceinline__ uint32_t pull_at(const A &a, const D &d) {       // less the own part
    if constexpr (A::kOne) return a.pull[I];
    else return a.pull[I] - (uint32_t)(cz_of(I) * d.Ps);       // (the members' planes differ)
}

// One cell (R float, at any plane) or the cells of planes z and z + 1 (R pf2, 1 <= z, z + 2 <
// nz: no periodic wrap between them) of a position.
template <int P, int WALL, int EXTRA, class R, class A, class D>
__device__ __forceinline__ void odd_cells(const A &a, const D &d, const int4 ci, uint32_t at, int z, bool trig, float st,
                                          float tx, float ty, float tz) {
    using PS = PairStorage<P>;
    using B = typename PS::B;
    constexpr bool TWO = std::is_same<R, pf2>::value;
    const uint32_t nb = (uint32_t)ci.y;
    const uint32_t col = (uint32_t)(ci.x & 0xFFFF) * (uint32_t)d.nx + ((uint32_t)ci.x >> 16);
    const int64_t plane = (int64_t)d.nx * d.ny;
    B *const base = static_cast<B *>(a.pops);
    // element read by direction i at plane z; the second cell's is one plane further
    auto index = [&](auto ic, uint32_t own) -> uint32_t {
        constexpr int i = decltype(ic)::value, cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
        uint32_t pull = pull_at<i>(a, d);
        if constexpr (!TWO && cz == 1) pull += z == 0 ? (uint32_t)d.nz * (uint32_t)d.Ps : 0u;
        if constexpr (!TWO && cz == -1) pull -= z == d.nz - 1 ? (uint32_t)d.nz * (uint32_t)d.Ps : 0u;
        if constexpr (cx == 0 && cy == 0) {
            return own + (own_at<i>(a, d) + pull);
        } else {
            const uint32_t f = (uint32_t)((int32_t)(nb << (31 - nbit(-cx, -cy))) >> 31);
            const uint32_t dx = (cy == 0 ? 0u : (uint32_t)(cy > 0 ? ci.z : ci.w)) - (uint32_t)cx;
            return (own + (f & dx)) + own_at<i>(a, d) + (f & pull);
        }
    };
    const uint32_t own = at + (uint32_t)z * (uint32_t)d.Ps;
    R v[Q];
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const uint32_t k = index(ic, own);
        if constexpr (TWO) v[i] = make_float2(PS::up1(base[k]), PS::up1(base[k + (uint32_t)d.Ps]));
        else v[i] = PS::up1(base[k]);
    });
    R gx = lit<R>(d.gf[0]), gy = lit<R>(d.gf[1]), gz = lit<R>(d.gf[2]);
    if (d.gz_field != nullptr) {
        const float *q = static_cast<const float *>(d.gz_field) + (plane * z + col);
        if constexpr (TWO) gz = add_(gz, make_float2(q[0], q[plane]));
        else gz = add_(gz, q[0]);
    }
    if (trig) {
        const float *zt = static_cast<const float *>(d.ztab) + z;
        R sc, ss;
        if constexpr (TWO) {
            sc = make_float2(mul_(st, zt[0]), mul_(st, zt[1]));
            ss = make_float2(mul_(st, zt[d.nz]), mul_(st, zt[d.nz + 1]));
        } else {
            sc = mul_(st, zt[0]);
            ss = mul_(st, zt[d.nz]);
        }
        gx = fma_(sc, lit<R>(tx), gx);
        gy = fma_(sc, lit<R>(ty), gy);
        gz = fma_(ss, lit<R>(tz), gz);
    }
    const float *tab = static_cast<const float *>(d.dtab) + (int64_t)col * 27;
    if constexpr (WALL == LBM_BOUZIDI) {
        if (nb != 0x1FFu)
            sfor<0, Q>([&](auto jc) {
                constexpr int j = decltype(jc)::value, cx = cx_of(j), cy = cy_of(j);
                if constexpr (cx != 0 || cy != 0)
                    if (!((nb >> nbit(cx, cy)) & 1u))
                        v[opp_of(j)] = fma_(lit<R>(tab[nbit(cx, cy) * 3 + 2]), v[j], v[opp_of(j)]);
            });
    }
    const MomentSums<R> ms = moment_sums<R, P == LBM_F32>(v);
    // the element a slot is written at is the one it was read at: the zero (which depends on
    // the data) keeps the compiler from carrying the addresses through the collision
    uint32_t bits;
    if constexpr (TWO) bits = __float_as_uint(ms.drho.x);
    else bits = __float_as_uint(ms.drho);
    const uint32_t wown = own + min(bits, a.zero);
    auto store = [&](auto ic, R f) {
        constexpr int ib = opp_of(decltype(ic)::value);
        const uint32_t k = index(std::integral_constant<int, ib>{}, wown);
        if constexpr (TWO) {
            base[k] = PS::down1(f.x);
            base[k + (uint32_t)d.Ps] = PS::down1(f.y);
        } else {
            base[k] = PS::down1(f);
        }
    };
    Macro<R> mm;
    if constexpr (WALL == LBM_BOUZIDI) {
        mm = pair_collide<P, false, R>(ms, gx, gy, gz, d.omegaf, a.f16_inv, a.f16_scale, nullptr,
                                       [&](auto ic, R f) { v[decltype(ic)::value] = f; });
        sfor<0, Q>([&](auto jc) {
            constexpr int j = decltype(jc)::value, cx = cx_of(j), cy = cy_of(j), kk = nbit(cx, cy);
            R f = v[j];
            if constexpr (cx != 0 || cy != 0)
                if (!((nb >> kk) & 1u))
                    f = fma_(lit<R>(tab[kk * 3]), f, mul_(lit<R>(tab[kk * 3 + 1]), v[opp_of(j)]));
            store(jc, f);
        });
    } else {
        R sk[5];
        mm = pair_collide<P, false, R>(ms, gx, gy, gz, d.omegaf, a.f16_inv, a.f16_scale,
                                       EXTRA == EX_MOMENTS ? sk : nullptr, store);
        if constexpr (EXTRA == EX_MOMENTS) {
            float *mo = static_cast<float *>(a.moments) + (own - (uint32_t)d.off);
            const R out[9] = {mm.rho, mm.ux, mm.uy, mm.uz, sk[0], sk[1], sk[2], sk[3], sk[4]};
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                float *q = mo + k * d.scells;
                if constexpr (TWO) {
                    q[0] = out[k].x;
                    q[d.Ps] = out[k].y;
                } else {
                    q[0] = out[k];
                }
            }
        }
    }
    if constexpr (EXTRA == EX_STATS) {
        double *s = a.stats + d.doff + plane * z + col;
        if constexpr (TWO) {
            add_stats(s, a.dstride, (double)mm.uz.x);
            add_stats(s + plane, a.dstride, (double)mm.uz.y);
        } else {
            add_stats(s, a.dstride, (double)mm.uz);
        }
    }
}

// Planes 1 .. nz - 2 in pairs, ZC / 2 pairs per thread (the table entry is read once for all);
// the first blocks take the planes that are left (0, nz - 1 and, for odd nz, nz - 2) singly.
template <int P, int WALL, int EXTRA, int BS, int MINB, int ZC, class A>
__global__ void __launch_bounds__(BS, MINB) k_odd2(const __grid_constant__ A a) {
    release_next_step();
    const PairTask tk = pair_task(a);
    const auto &d = pair_member(a, tk.m);
    uint32_t nb_plane, zg;
    if constexpr (A::kOne) {
        nb_plane = a.nb_plane;
        zg = fastdiv(tk.local, a.nb_mul, a.nb_shr);
    } else {
        nb_plane = a.nb_plane[tk.m];
        zg = fastdiv(tk.local, a.nb_mul[tk.m], a.nb_shr[tk.m]);
    }
    const uint32_t r = (tk.local - zg * nb_plane) * BS + threadIdx.x;
    if (r >= (uint32_t)d.Ps) return;
    const int4 ci = d.cellinfo[r];
    if (ci.x == -1) return;
    const bool trig = d.trig && pair_t(a) < d.t_end;
    float st = 0, tx = 0, ty = 0, tz = 0;
    if (trig) {
        st = pair_st(a, tk.m);
        const float *ft = static_cast<const float *>(d.ftabc) + r;
        tx = ft[0];
        ty = ft[d.Ps];
        tz = ft[2 * (uint32_t)d.Ps];
    }
    await_previous_step();
    const int singles = odd_single_planes(d.nz);
    if ((int)zg < singles) {
        const int z = zg == 0 ? 0 : d.nz - (int)zg;
        odd_cells<P, WALL, EXTRA, float>(a, d, ci, (uint32_t)d.off + r, z, trig, st, tx, ty, tz);
        return;
    }
#pragma unroll 1
    for (int k = 0; k < ZC / 2; ++k) {
        const int z = 1 + ((int)zg - singles) * ZC + 2 * k;
        if (z + 2 >= d.nz) break;
        uint32_t at = (uint32_t)d.off + r;
        int4 cj = ci;
        asm volatile("" : "+r"(at), "+r"(cj.x), "+r"(cj.y), "+r"(cj.z), "+r"(cj.w));    // nothing of a pass outlives it
        odd_cells<P, WALL, EXTRA, pf2>(a, d, cj, at, z, trig, st, tx, ty, tz);
    }
}

}  // namespace lbm

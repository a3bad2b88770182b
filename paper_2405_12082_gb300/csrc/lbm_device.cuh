// lbm_device.cuh -- device building blocks of the D3Q27 MRT step.
//
// * Lattice (Appendix A): velocity order, opposite directions, weights.
// * Storage traits: populations are stored as f_i - w_i in double, float, half
//   (scaled by 2^s) or bfloat16; arithmetic runs in double or float.
// * The single-buffer AA access pattern: an even step reads and writes the cell's
//   own slots (slot i read as f_i, f*_i written to slot ibar); an odd step pulls
//   f_i from slot ibar of x - c_i and pushes f*_i to slot i of x + c_i.  Both touch
//   each slot exactly once, so the update is in place and race-free.  Wall links
//   (x - c_i solid) read and write the cell's own slot instead, which realises
//   half-way bounce-back; Bouzidi links add the interpolation of Eqs. (fbc1)-(fbc2)
//   on top of the same slots.
// * The collision of Eqs. (collision), (m*), (k*f*) in closed form.  With Lambda =
//   diag[1,1,1,1,omega x5,1 x18] every non-shear moment leaves the collision at
//   m^eq + R/2, so f* = f^eq + (1/2) g . grad_u f^eq + (1 - omega) sum_{k=4..8} C_k
//   (m_k - m_k^eq + R_k / 2), where C_k is column k of (M^T)^{-1} (nonzero only on
//   the 4 or 6 populations with the matching second-order velocity product).  The
//   sixth-order Hermite equilibrium factorises on D3Q27 as rho w_i psi(c_ix, u_x)
//   psi(c_iy, u_y) psi(c_iz, u_z), psi(0,u)/psi(0,0) = 1 - 3u^2/2 and
//   psi(+-1,u)/psi(+-1,0) = 1 +- 3u + 3u^2, which is what is evaluated.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <type_traits>

#include "lbm.h"

namespace lbm {

// ---- lattice, Appendix A ----------------------------------------------------------
constexpr int Q = 27;
__host__ __device__ constexpr int cx_of(int i) {
    constexpr int v[27] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1};
    return v[i];
}
__host__ __device__ constexpr int cy_of(int i) {
    constexpr int v[27] = {0, 0, 0, 1, -1, 0, 0, 1, 1, -1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, 1, -1, -1, 1, 1, -1, -1};
    return v[i];
}
__host__ __device__ constexpr int cz_of(int i) {
    constexpr int v[27] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, 1, -1, -1, 1, 1, -1, -1, 1, 1, 1, 1, -1, -1, -1, -1};
    return v[i];
}
__host__ __device__ constexpr int opp_of(int i) {
    for (int j = 0; j < 27; ++j)
        if (cx_of(j) == -cx_of(i) && cy_of(j) == -cy_of(i) && cz_of(j) == -cz_of(i)) return j;
    return -1;
}
// Eq. (omegas): w0 = 8/27, w0/4 on faces, w0/16 on edges, w0/64 on corners.
__host__ __device__ constexpr double w_of(int i) {
    return i == 0 ? 8.0 / 27.0 : (i <= 6 ? 2.0 / 27.0 : (i <= 18 ? 1.0 / 54.0 : 1.0 / 216.0));
}
// index of the velocity (cx, cy, cz)
__host__ __device__ constexpr int dir_of(int cx, int cy, int cz) {
    for (int j = 0; j < 27; ++j)
        if (cx_of(j) == cx && cy_of(j) == cy && cz_of(j) == cz) return j;
    return -1;
}
// in-plane neighbourhood bit of (cx, cy): bit (cy + 1) * 3 + (cx + 1)
__host__ __device__ constexpr int nbit(int cx, int cy) { return (cy + 1) * 3 + (cx + 1); }

template <int I, int N, class F>
__device__ __forceinline__ void sfor(F &&f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        sfor<I + 1, N>(f);
    }
}

// Row k of the moment basis of Eq. (Mmatrix) at velocity i: m_k = sum_i mt_coef(k, i) f_i.
__host__ __device__ constexpr int mt_coef(int k, int i) {
    const int x = cx_of(i), y = cy_of(i), z = cz_of(i);
    const int x2 = x * x, y2 = y * y, z2 = z * z;
    switch (k) {
        case 0: return 1;
        case 1: return x;
        case 2: return y;
        case 3: return z;
        case 4: return x * y;
        case 5: return x * z;
        case 6: return y * z;
        case 7: return x2 - y2;
        case 8: return x2 - z2;
        case 9: return x2 + y2 + z2;
        case 10: return x * y2 + x * z2;
        case 11: return x2 * y + y * z2;
        case 12: return x2 * z + y2 * z;
        case 13: return x * y2 - x * z2;
        case 14: return x2 * y - y * z2;
        case 15: return x2 * z - y2 * z;
        case 16: return x * y * z;
        case 17: return x2 * y2 + x2 * z2 + y2 * z2;
        case 18: return x2 * y2 + x2 * z2 - y2 * z2;
        case 19: return x2 * y2 - x2 * z2;
        case 20: return x2 * y * z;
        case 21: return x * y2 * z;
        case 22: return x * y * z2;
        case 23: return x * y2 * z2;
        case 24: return x2 * y * z2;
        case 25: return x2 * y2 * z;
        default: return x2 * y2 * z2;
    }
}

// (M^T)^{-1}, the back transform of Eq. (k*f*), by Gauss-Jordan elimination with
// partial pivoting, evaluated by the compiler: a[i][k] is the weight of moment k in
// population i.
struct MtInverse { double a[27][27]; };
constexpr MtInverse make_mt_inverse() {
    double A[27][54] = {};
    for (int k = 0; k < 27; ++k) {
        for (int i = 0; i < 27; ++i) A[k][i] = (double)mt_coef(k, i);
        A[k][27 + k] = 1.0;
    }
    for (int col = 0; col < 27; ++col) {
        int piv = col;
        for (int r = col + 1; r < 27; ++r) {
            const double a = A[r][col] < 0 ? -A[r][col] : A[r][col];
            const double b = A[piv][col] < 0 ? -A[piv][col] : A[piv][col];
            if (a > b) piv = r;
        }
        for (int j = 0; j < 54; ++j) {
            const double t = A[col][j];
            A[col][j] = A[piv][j];
            A[piv][j] = t;
        }
        const double d = A[col][col];
        for (int j = 0; j < 54; ++j) A[col][j] /= d;
        for (int r = 0; r < 27; ++r) {
            if (r == col || A[r][col] == 0.0) continue;
            const double fct = A[r][col];
            for (int j = 0; j < 54; ++j) A[r][j] -= fct * A[col][j];
        }
    }
    MtInverse out{};
    for (int i = 0; i < 27; ++i)
        for (int k = 0; k < 27; ++k) {
            const double v = A[i][27 + k];
            out.a[i][k] = (v < 1e-14 && v > -1e-14) ? 0.0 : v;    // exact zeros of the inverse
        }
    return out;
}
constexpr MtInverse kMtInv = make_mt_inverse();

// ---- arithmetic ------------------------------------------------------------------------
// The collision is written in single-rounding operations (no contraction left to the
// compiler), so every kernel that runs it -- one cell per thread, two cells per thread on
// the paired FP32 instructions, staged -- produces the same bits.  pf2 is a pair of cells
// in one 64-bit register pair: one FFMA2 / FADD2 / FMUL2 does both cells' operation in one
// issue slot (the same FP32 lane rate as two scalar instructions, half the issue slots).
using pf2 = float2;
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float neg_(float a) { return -a; }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double neg_(double a) { return -a; }
__device__ __forceinline__ pf2 fma_(pf2 a, pf2 b, pf2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ pf2 mul_(pf2 a, pf2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ pf2 add_(pf2 a, pf2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ pf2 sub_(pf2 a, pf2 b) { return fma_(b, make_float2(-1.f, -1.f), a); }   // same rounding
__device__ __forceinline__ pf2 neg_(pf2 a) { return make_float2(-a.x, -a.y); }
// a + b where a term is a rounded product: on pairs the compiler fuses an addition with the
// product before it, on single cells it does not.
__device__ __forceinline__ float sum_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double sum_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ pf2 sum_(pf2 a, pf2 b) { return fma_(a, make_float2(1.f, 1.f), b); }

// The scalar type of R and a constant of type R.
template <class R> struct scalar_of { using type = R; };
template <> struct scalar_of<pf2> { using type = float; };
template <class R> __device__ __forceinline__ R lit(typename scalar_of<R>::type c) {
    if constexpr (std::is_same<R, pf2>::value) return make_float2(c, c);
    else return c;
}

// 1 / x.  FP32: the hardware's approximate reciprocal (within one unit in the last place) and one
// Newton-Raphson iteration r + r (1 - x r) on fused multiply-adds, which rounds correctly from
// there (Markstein 1990) but for x whose mantissa is all ones: the division's result in three
// instructions and without its branch (F16S, R = 96 pipe: 804 us per step, with the division 849).
__device__ __forceinline__ float recip_(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return __fmaf_rn(r, __fmaf_rn(-x, r, 1.f), r);
}
__device__ __forceinline__ double recip_(double x) { return 1.0 / x; }
__device__ __forceinline__ pf2 recip_(pf2 x) { return make_float2(recip_(x.x), recip_(x.y)); }

// ---- storage ------------------------------------------------------------------------
// ld / st convert between the stored value and f - w; ldr / str move the stored value
// unscaled (the step kernels of the scaled half format work in units of 2^-s, see collide).
template <int P> struct Storage;
template <> struct Storage<LBM_F64> {
    using T = double; using R = double;
    static constexpr bool kScaled = false;
    static __device__ __forceinline__ R ld(const T *p, R) { return *p; }
    static __device__ __forceinline__ void st(T *p, R v, R) { *p = v; }
    static __device__ __forceinline__ R ldr(const T *p) { return *p; }
    static __device__ __forceinline__ void str(T *p, R v) { *p = v; }
};
template <> struct Storage<LBM_F32> {
    using T = float; using R = float;
    static constexpr bool kScaled = false;
    static __device__ __forceinline__ R ld(const T *p, R) { return *p; }
    static __device__ __forceinline__ void st(T *p, R v, R) { *p = v; }
    static __device__ __forceinline__ R ldr(const T *p) { return *p; }
    static __device__ __forceinline__ void str(T *p, R v) { *p = v; }
};
template <> struct Storage<LBM_F16S> {
    using T = __half; using R = float;
    static constexpr bool kScaled = true;
    static __device__ __forceinline__ R ld(const T *p, R inv_scale) { return __half2float(*p) * inv_scale; }
    static __device__ __forceinline__ void st(T *p, R v, R scale) { *p = __float2half_rn(v * scale); }
    static __device__ __forceinline__ R ldr(const T *p) { return __half2float(*p); }
    static __device__ __forceinline__ void str(T *p, R v) { *p = __float2half_rn(v); }
};
template <> struct Storage<LBM_BF16> {
    using T = __nv_bfloat16; using R = float;
    static constexpr bool kScaled = false;
    static __device__ __forceinline__ R ld(const T *p, R) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void st(T *p, R v, R) { *p = __float2bfloat16_rn(v); }
    static __device__ __forceinline__ R ldr(const T *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void str(T *p, R v) { *p = __float2bfloat16_rn(v); }
};

// ---- per-member description (host fills, device reads) ---------------------------------
// Storage layouts.  Dense: every cell of the box is stored, index (z ny + y) nx + x.
// Compact (pipes with half-way or Bouzidi walls): each row (y, z) stores only its run
// of fluid cells x0(y) .. x0(y) + span(y) - 1, starting on a 64-byte boundary; a plane
// holds Ps elements and cell (x, y, z) sits at z Ps + rowbase(y) + x - x0(y).  Solid
// cells have no storage (those walls never touch them), so every DRAM access atom
// carries fluid data except at the end of a row, and threads map onto stored cells only.
struct Member {
    int32_t nx, ny, nz, geometry;
    int64_t off;        // first stored cell of this member inside each population plane
    int64_t cells;      // nx * ny * nz
    int64_t scells;     // stored cells: cells (dense) or nz * Ps (compact)
    int64_t doff;       // first cell of this member in dense per-cell arrays (statistics)
    int32_t compact, Ps;
    uint32_t ps_mul, ps_shr;   // magic division by Ps
    const int32_t *rowbase;    // compact: [ny] start of row y inside a plane
    const int32_t *rowx0;      // compact: [ny] first fluid x of row y
    const uint16_t *rowof;     // compact: [Ps] row of each stored position (0xFFFF: padding)
    const int4 *cellinfo;      // compact: [Ps] per stored position: y | x << 16 (all ones:
                               // padding), the column's fluid mask, and the storage offsets
                               // of the rows y - 1 and y + 1 at the same x
    int64_t block0;     // first block of this member in a flat launch
    int64_t n_fluid;
    int64_t d2max;      // pipe: fluid iff (2x-nx+1)^2 + (2y-ny+1)^2 <= d2max
    double R, omega;
    double g[3];
    // trigger force, Eq. (TurbForce)
    int32_t trig, n_modes, kz, pad0;
    int32_t k_theta[LBM_MAX_TRIGGER_MODES];
    double amp[LBM_MAX_TRIGGER_MODES];     // h * A0 * weight
    double cph[LBM_MAX_TRIGGER_MODES], sph[LBM_MAX_TRIGGER_MODES];
    double kappa, l0, l, period;
    int64_t t_end;
    const void *gz_field;
    uint32_t nx_mul, nx_shr, ny_mul, ny_shr;   // magic division by nx and ny
    float gf[3], omegaf;       // float copies of g and omega for the FP32 kernels
    // general relaxation matrix Lambda = diag(lambda_k): 1 - lambda_k for k = 4..26
    // (k = 0..3 are conserved; read only by the general-rates collision)
    double om1k[23];
    float om1kf[23];
    const uint16_t *colmask;   // [ny][nx] in-plane 3x3 fluid mask of every column (device)
    const void *ftab;          // trigger: [3][ny][nx] column factors (P_x, P_y, P_z), compute type
    const void *ztab;          // trigger: [2][nz] cos, sin of kz 2 pi z / L, compute type
    const void *dtab;          // Bouzidi walls: [ny][nx][9][3] coefficients A, B, C of the link
                               // (cx, cy) at index nbit(cx, cy), compute type
    const int32_t *fluidcol;   // dense pipe: [Pw] dense columns y nx + x of the fluid cells
    int32_t Pw;                // positions of a plane that threads map to: the fluid columns of a
                               // dense pipe, else Ps
    uint32_t pw_mul, pw_shr;   // magic division by Pw
    const uint32_t *pairinfo;  // compact: [Ps / 2] per pair of stored positions (see PAIR_*)
    const void *ftabc;         // trigger, compact: [3][Ps] column factors by stored position
    const int4 *sg[2];         // compact: row groups of the two staged launch shapes (2 int4
                               // per group, see lbm_staged.cuh), nsg[k] groups (0: shape
                               // not available for this member)
    int32_t nsg[2];
};

// An entry of pairinfo: whether the first and the second position are fluid cells, whether
// one of them has a wall link, and the dense column y nx + x of the first.
constexpr uint32_t PAIR_A = 1, PAIR_B = 2, PAIR_WALL = 4;
constexpr int PAIR_SHIFT = 3;

// Unsigned division by a fixed divisor d >= 1 for n < 2^31 (Granlund-Montgomery with
// a 31-bit dividend): l = ceil(log2 d), mul = ceil(2^(31+l) / d) < 2^32, and
// n / d = umulhi(n, mul) >> (l - 1).  d = 1 is flagged by shr = 0xFFFFFFFF.
inline void fastdiv_setup(uint32_t d, uint32_t &mul, uint32_t &shr) {
    if (d <= 1) { mul = 0; shr = 0xFFFFFFFFu; return; }
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    const uint64_t m = ((1ull << (31 + l)) + d - 1) / d;
    mul = (uint32_t)m;
    shr = l - 1;
}
__device__ __forceinline__ uint32_t fastdiv(uint32_t n, uint32_t mul, uint32_t shr) {
    return shr == 0xFFFFFFFFu ? n : (__umulhi(n, mul) >> shr);
}

// Per-step values for graph-captured chunks of steps: step index and sin(2 pi t / T) of
// every member's trigger (0 when off), filled by the host before each replay.
struct StepTime {
    int64_t t;
    double st[LBM_MAX_MEMBERS];
    float stf[LBM_MAX_MEMBERS];
};

struct StepArgs {
    void *pops;               // [27][stride] storage elements
    int64_t stride;           // cells per population plane (all members)
    const Member *members;    // device array
    int32_t n_members;
    int32_t nblocks_total;
    int64_t t;                // index of the step being taken
    float f16_scale, f16_inv;
    double *stats;            // [4][dstride] FP64 accumulators (sample steps), dense cells
    int64_t dstride;          // cells of all members in dense per-cell arrays
    double st[LBM_MAX_MEMBERS];      // sin(2 pi t / T) per member (0 when off)
    float stf[LBM_MAX_MEMBERS];      // the same in float for the FP32 kernels
    int32_t block0[LBM_MAX_MEMBERS + 1];
    const StepTime *times;    // when set, t and st come from times[tidx] (graph replays)
    int32_t tidx;
    void *moments;            // adjoint recompute: [9][cells] rho, u, s4..s8 of member 0
    int32_t collision;        // collision model (MODEL_* bits), the same for every member
    uint32_t zero;            // 0 (see store_pops)
    int32_t overlap;          // the kernel may start while the step before it drains
    int32_t single;           // a shape of several planes per thread runs one (small contexts)
    int32_t pairs;            // the step runs on pairs of cells (lbm_pair.cuh)
    int32_t stage_cap;        // staged shapes: storage elements per direction segment
    int32_t sg_sel;           // staged shapes: which row-group table (0 or 1)
    int32_t *err;             // device status word (bounded waits that expired), or NULL
    int32_t skip_tile;        // failure-detection tests: a staged tile whose copies are never
                              // issued (its wait expires); -1 otherwise
};

__device__ __forceinline__ int find_member(const StepArgs &a, int blk) {
    int lo = 0, hi = a.n_members - 1;
    while (lo < hi) {          // largest m with block0[m] <= blk
        int mid = (lo + hi + 1) >> 1;
        if (a.block0[mid] <= blk) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---- geometry --------------------------------------------------------------------------
struct CellPos {
    int x, y, z;
    int32_t lc;              // storage index inside the member
    int32_t di;              // dense index (z ny + y) nx + x inside the member
    int32_t ox[3], oy[3], oz[3]; // neighbour offsets for c = -1, 0, +1 (periodic)
    uint32_t nb;             // in-plane fluid mask of the 3x3 neighbourhood
};

// Fluid test of a column (x, y) (pipe: distance to the axis < R, see lbm.h).
__host__ __device__ __forceinline__ bool col_fluid(const Member &d, int x, int y) {
    if (d.geometry == LBM_BOX) return true;
    const int64_t X = 2 * (int64_t)x - d.nx + 1, Y = 2 * (int64_t)y - d.ny + 1;
    return X * X + Y * Y <= d.d2max;
}

// Neighbour offsets (storage units) for c = -1, 0, +1 along x, y and z.
__device__ __forceinline__ void cell_offsets(const Member &d, CellPos &p) {
    if (!d.compact) {
        const int32_t nx = d.nx, nxy = d.nx * d.ny;
        p.ox[0] = p.x == 0 ? nx - 1 : -1;
        p.ox[1] = 0;
        p.ox[2] = p.x == nx - 1 ? -(nx - 1) : 1;
        p.oy[0] = p.y == 0 ? (d.ny - 1) * nx : -nx;
        p.oy[1] = 0;
        p.oy[2] = p.y == d.ny - 1 ? -(d.ny - 1) * nx : nx;
        p.oz[0] = p.z == 0 ? (d.nz - 1) * nxy : -nxy;
        p.oz[1] = 0;
        p.oz[2] = p.z == d.nz - 1 ? -(d.nz - 1) * nxy : nxy;
    } else {
        // rows of a pipe never reach the box edge: no x or y wrap.  A neighbour row
        // without fluid gets an unused offset (its cells are solid in the mask).
        const int32_t me = d.rowbase[p.y] - d.rowx0[p.y];
        p.ox[0] = -1;
        p.ox[1] = 0;
        p.ox[2] = 1;
        p.oy[0] = p.y > 0 ? (d.rowbase[p.y - 1] - d.rowx0[p.y - 1]) - me : 0;
        p.oy[1] = 0;
        p.oy[2] = p.y < d.ny - 1 ? (d.rowbase[p.y + 1] - d.rowx0[p.y + 1]) - me : 0;
        p.oz[0] = p.z == 0 ? (d.nz - 1) * d.Ps : -d.Ps;
        p.oz[1] = 0;
        p.oz[2] = p.z == d.nz - 1 ? -(d.nz - 1) * d.Ps : d.Ps;
    }
}

// Cell of storage index sidx (< scells) of member d.  Returns whether it is a fluid cell;
// for a compact padding slot nothing else is set.
__device__ __forceinline__ bool cell_from_storage(const Member &d, uint32_t sidx, CellPos &p) {
    if (!d.compact) {
        const uint32_t q = fastdiv(sidx, d.nx_mul, d.nx_shr);
        p.x = (int)(sidx - q * (uint32_t)d.nx);
        p.z = (int)fastdiv(q, d.ny_mul, d.ny_shr);
        p.y = (int)(q - (uint32_t)p.z * (uint32_t)d.ny);
        p.lc = (int32_t)sidx;
        p.di = (int32_t)sidx;
    } else {
        // one 16-byte table load gives position, fluid mask and row offsets, so the
        // neighbour addresses of the odd step wait on a single load
        p.z = (int)fastdiv(sidx, d.ps_mul, d.ps_shr);
        const int32_t r = (int32_t)(sidx - (uint32_t)p.z * (uint32_t)d.Ps);
        const int4 ci = d.cellinfo[r];
        if (ci.x == -1) return false;
        p.y = ci.x & 0xFFFF;
        p.x = (int)((uint32_t)ci.x >> 16);
        p.lc = (int32_t)sidx;
        p.di = (p.z * d.ny + p.y) * d.nx + p.x;
        p.nb = (uint32_t)ci.y;
        p.ox[0] = -1;
        p.ox[1] = 0;
        p.ox[2] = 1;
        p.oy[0] = ci.z;
        p.oy[1] = 0;
        p.oy[2] = ci.w;
        p.oz[0] = p.z == 0 ? (d.nz - 1) * d.Ps : -d.Ps;
        p.oz[1] = 0;
        p.oz[2] = p.z == d.nz - 1 ? -(d.nz - 1) * d.Ps : d.Ps;
        return (p.nb >> 4) & 1u;
    }
    p.nb = d.colmask[p.y * d.nx + p.x];
    cell_offsets(d, p);
    return (p.nb >> 4) & 1u;
}

// Cell of thread index `local` of a launch over Pw positions x plane groups of zc planes (the
// first plane of its group): the fluid columns of a dense pipe are packed, so its warps hold
// fluid cells only.  Returns whether there is a fluid cell.
__device__ __forceinline__ bool cell_from_work(const Member &d, uint32_t local, uint32_t zc, CellPos &p) {
    const uint32_t g = fastdiv(local, d.pw_mul, d.pw_shr);
    const uint32_t z = g * zc;
    if (z >= (uint32_t)d.nz) return false;
    const uint32_t r = local - g * (uint32_t)d.Pw;
    if (d.fluidcol == nullptr) return cell_from_storage(d, z * (uint32_t)d.Ps + r, p);
    const uint32_t col = (uint32_t)d.fluidcol[r];
    p.y = (int)fastdiv(col, d.nx_mul, d.nx_shr);
    p.x = (int)(col - (uint32_t)p.y * (uint32_t)d.nx);
    p.z = (int)z;
    p.lc = p.di = (int32_t)(z * (uint32_t)d.Ps + col);
    p.nb = d.colmask[col];
    cell_offsets(d, p);
    return true;
}

// Cell of dense index di (< cells).  p.lc is the storage index of a fluid cell (every
// cell in the dense layout); returns whether the cell is fluid.
__device__ __forceinline__ bool cell_from_dense(const Member &d, uint32_t di, CellPos &p) {
    const uint32_t q = fastdiv(di, d.nx_mul, d.nx_shr);
    p.x = (int)(di - q * (uint32_t)d.nx);
    p.z = (int)fastdiv(q, d.ny_mul, d.ny_shr);
    p.y = (int)(q - (uint32_t)p.z * (uint32_t)d.ny);
    p.di = (int32_t)di;
    p.nb = d.colmask[p.y * d.nx + p.x];
    const bool fluid = (p.nb >> 4) & 1u;
    if (!d.compact) p.lc = (int32_t)di;
    else p.lc = fluid ? p.z * d.Ps + d.rowbase[p.y] + (p.x - d.rowx0[p.y]) : -1;
    cell_offsets(d, p);
    return fluid;
}

template <int I>
__device__ __forceinline__ int32_t nb_offset(const CellPos &p) {   // x + c_I
    return p.ox[cx_of(I) + 1] + p.oy[cy_of(I) + 1] + p.oz[cz_of(I) + 1];
}
template <int I>
__device__ __forceinline__ int32_t src_offset(const CellPos &p) {  // x - c_I
    return p.ox[1 - cx_of(I)] + p.oy[1 - cy_of(I)] + p.oz[1 - cz_of(I)];
}
template <int I>
__device__ __forceinline__ bool src_is_fluid(const CellPos &p) {
    return (p.nb >> nbit(-cx_of(I), -cy_of(I))) & 1u;
}
template <int I>
__device__ __forceinline__ bool dst_is_fluid(const CellPos &p) {
    return (p.nb >> nbit(cx_of(I), cy_of(I))) & 1u;
}

// ---- Bouzidi link coefficients, Eqs. (fbc1)-(fbc2) ---------------------------------------
// For a wall-pointing direction J of a fluid cell (x + c_J solid), the population
// returning in direction Jbar is A f*_J(x) + B f*_Jbar(x) + C f*_J(x - c_J).
template <class R>
struct BLink { R A, B, C; };

// The coefficients come from a per-column table filled on the host in FP64 from Delta,
// the fraction of the link from x to the circle r = R (the wall is a cylinder, so they
// depend on (x, y) and (cx, cy) only): Delta >= 1/2: A = 1 / (2 Delta), B = (2 Delta - 1) /
// (2 Delta), C = 0; Delta < 1/2 with x - c_J fluid: A = 2 Delta, B = 0, C = 1 - 2 Delta;
// otherwise the half-way values A = 1, B = C = 0.
template <class R, int J>
__device__ __forceinline__ BLink<R> bouzidi_link(const Member &d, const CellPos &p) {
    constexpr int cx = cx_of(J), cy = cy_of(J);
    const R *tab = static_cast<const R *>(d.dtab);
    const int64_t k = ((int64_t)(p.y * d.nx + p.x) * 9 + nbit(cx, cy)) * 3;
    return BLink<R>{tab[k], tab[k + 1], tab[k + 2]};
}

// The slot of a wall-pointing direction J holds A f*_J + B f*_Jbar of the previous step;
// the read of direction Jbar adds C f*_J(x - c_J), which is the value just read for J.
template <class R>
__device__ __forceinline__ void bouzidi_load_fix(const Member &d, const CellPos &p, R (&v)[27]) {
    if (p.nb == 0x1FFu) return;
    sfor<0, 27>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        if constexpr (cx_of(j) != 0 || cy_of(j) != 0) {
            if (!dst_is_fluid<j>(p)) {
                BLink<R> b = bouzidi_link<R, j>(d, p);
                v[opp_of(j)] = fma_(b.C, v[j], v[opp_of(j)]);
            }
        }
    });
}

// ---- loading and storing the 27 populations of a cell ------------------------------------
// PAR 0: natural layout (after an odd step); PAR 1: reversed layout (after an even step).
// Slot of direction i read at a cell: PAR 0 -> (i, x); PAR 1 -> (ibar, x - c_i), or (i, x)
// across a wall link.  Slot written: PAR 0 -> (ibar, x); PAR 1 -> (i, x + c_i), or (ibar, x)
// across a wall link.  Wall links choose the address with a select, not a branch.
// Element indices are 32-bit: the library keeps 27 x stride below 2^32.
// RAW: the values stay in storage units (only the step kernels, see collide).
template <int P, bool RAW>
__device__ __forceinline__ typename Storage<P>::R ld_pop(const typename Storage<P>::T *q, typename Storage<P>::R inv) {
    if constexpr (RAW) return Storage<P>::ldr(q);
    else return Storage<P>::ld(q, inv);
}
template <int P, bool RAW>
__device__ __forceinline__ void st_pop(typename Storage<P>::T *q, typename Storage<P>::R v, typename Storage<P>::R sc) {
    if constexpr (RAW) Storage<P>::str(q, v);
    else Storage<P>::st(q, v, sc);
}

template <int P, int PAR, int WALL, bool RAW = false>
__device__ __forceinline__ void load_pops(const StepArgs &a, const Member &d, const CellPos &p,
                                          typename Storage<P>::R (&v)[Q]) {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const T *base = static_cast<const T *>(a.pops) + d.off;
    const uint32_t st = (uint32_t)a.stride;
    const uint32_t lc = (uint32_t)p.lc;
    const R inv = (R)a.f16_inv;
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int ib = opp_of(i);
        if constexpr (PAR == 0) {
            v[i] = ld_pop<P, RAW>(base + (i * st + lc), inv);
        } else {
            const uint32_t pull = ib * st + (uint32_t)(p.lc + src_offset<i>(p));
            if constexpr (WALL == LBM_FULLWAY || (cx_of(i) == 0 && cy_of(i) == 0)) {
                v[i] = ld_pop<P, RAW>(base + pull, inv);
            } else {
                const uint32_t own = i * st + lc;
                v[i] = ld_pop<P, RAW>(base + (src_is_fluid<i>(p) ? pull : own), inv);
            }
        }
    });
    if constexpr (WALL == LBM_BOUZIDI) bouzidi_load_fix<R>(d, p, v);
}

template <int P, int PAR, int WALL, bool RAW = false>
__device__ __forceinline__ void store_pops(const StepArgs &a, const Member &d, const CellPos &p,
                                           typename Storage<P>::R (&v)[Q]) {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    // a slot is written where it was read: the zero keeps the compiler from carrying the 27
    // addresses through the collision in registers
    T *base = static_cast<T *>(a.pops) + d.off + a.zero;
    const uint32_t st = (uint32_t)a.stride + a.zero;
    const uint32_t lc = (uint32_t)p.lc + a.zero;
    const R sc = (R)a.f16_scale;
    if constexpr (WALL == LBM_BOUZIDI) {
        // the value reflected into slot Jbar becomes A f*_J + B f*_Jbar
        if (p.nb != 0x1FFu) {
            R out[Q];
            sfor<0, Q>([&](auto ic) { constexpr int i = decltype(ic)::value; out[i] = v[i]; });
            sfor<0, Q>([&](auto jc) {
                constexpr int j = decltype(jc)::value;
                if constexpr (cx_of(j) != 0 || cy_of(j) != 0) {
                    if (!dst_is_fluid<j>(p)) {
                        BLink<R> b = bouzidi_link<R, j>(d, p);
                        out[j] = fma_(b.A, v[j], mul_(b.B, v[opp_of(j)]));
                    }
                }
            });
            sfor<0, Q>([&](auto ic) { constexpr int i = decltype(ic)::value; v[i] = out[i]; });
        }
    }
    sfor<0, Q>([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int ib = opp_of(i);
        if constexpr (PAR == 0) {
            st_pop<P, RAW>(base + (ib * st + lc), v[i], sc);
        } else {
            const uint32_t push = i * st + (lc + (uint32_t)nb_offset<i>(p));
            if constexpr (WALL == LBM_FULLWAY || (cx_of(i) == 0 && cy_of(i) == 0)) {
                st_pop<P, RAW>(base + push, v[i], sc);
            } else {
                const uint32_t own = ib * st + lc;
                st_pop<P, RAW>(base + (dst_is_fluid<i>(p) ? push : own), v[i], sc);
            }
        }
    });
}

// ---- acceleration g(x, t), Sec. II.B ----------------------------------------------------------
// The trigger force of Eq. (TurbForce) factorises into st(t) x z-factor x column factor:
// g_x = st cos(2 pi kz z / L) P_x(x, y), g_y = st cos(...) P_y(x, y),
// g_z = st sin(2 pi kz z / L) P_z(x, y); the column factors (zero outside the radial
// band) and the z factors are tabulated once per force by k_force_tables.
// Member parameters in the compute type (no FP64 arithmetic or conversion in FP32 kernels).
template <class R> __device__ __forceinline__ R g_of(const Member &d, int k) {
    if constexpr (sizeof(R) == 4) return d.gf[k]; else return d.g[k];
}
template <class R> __device__ __forceinline__ const R *lam1_of(const Member &d) {
    if constexpr (sizeof(R) == 4) return d.om1kf;
    else return d.om1k;
}
template <class R> __device__ __forceinline__ R omega_of(const Member &d) {
    if constexpr (sizeof(R) == 4) return d.omegaf; else return d.omega;
}
// sin(2 pi t / T) of member m for this step, in the compute type.
template <class R> __device__ __forceinline__ R st_of(const StepArgs &a, int m) {
    if constexpr (sizeof(R) == 4) return a.times ? a.times[a.tidx].stf[m] : a.stf[m];
    else return a.times ? a.times[a.tidx].st[m] : a.st[m];
}

template <class R>
__device__ __forceinline__ void acceleration(const Member &d, const CellPos &p, int64_t t, R st,
                                             R &gx, R &gy, R &gz) {
    gx = g_of<R>(d, 0);
    gy = g_of<R>(d, 1);
    gz = g_of<R>(d, 2);
    if (d.gz_field != nullptr) gz += static_cast<const R *>(d.gz_field)[p.di];
    if (d.trig && t < d.t_end) {
        const R *ft = static_cast<const R *>(d.ftab);
        const R *zt = static_cast<const R *>(d.ztab);
        const int32_t col = p.y * d.nx + p.x, ncol = d.nx * d.ny;
        const R sc = mul_(st, zt[p.z]), ss = mul_(st, zt[d.nz + p.z]);
        gx = fma_(sc, ft[col], gx);
        gy = fma_(sc, ft[ncol + col], gy);
        gz = fma_(ss, ft[2 * ncol + col], gz);
    }
}

// Column and z factors of the trigger force (see acceleration), in double.
__device__ __forceinline__ void trigger_column(const Member &d, int x, int y, double &Px, double &Py, double &Pz) {
    Px = Py = Pz = 0.0;
    if (d.geometry != LBM_PIPE || !d.trig) return;
    const double px = 0.5 * (double)(2 * x - d.nx + 1), py = 0.5 * (double)(2 * y - d.ny + 1);
    const double r = sqrt(px * px + py * py);
    const double R = d.R, l0 = d.l0, l = d.l, L = (double)d.nz;
    if (!(r >= R - l0 - l && r <= R - l0 && r > 0.0)) return;
    const double ir = 1.0 / r, ct = px * ir, sn = py * ir;
    double sa, ca;
    sincospi(2.0 * (R - r - l0) / l, &sa, &ca);
    const double kz = (double)d.kz, kap = d.kappa;
    const double twopi = 6.283185307179586476925286766559;
    double Ar = 0, At = 0, Az = 0;
    for (int q = 0; q < d.n_modes; ++q) {
        const int kt = d.k_theta[q];
        double ck = 1, sk = 0;           // cos, sin of kt theta by repeated rotation
        for (int k = 0; k < kt; ++k) {
            const double c2 = ck * ct - sk * sn;
            sk = sk * ct + ck * sn;
            ck = c2;
        }
        const double cang = ck * d.cph[q] - sk * d.sph[q];
        const double sang = sk * d.cph[q] + ck * d.sph[q];
        const double A = d.amp[q];
        Ar += A * kap * (R * ir) * (kz * l / L) * (1.0 - ca) * cang;   // F_r = -st cz Ar
        At += A * (1.0 - kap) * (kz / kt) * (twopi * R / L) * sa * sang; // F_t =  st cz At
        Az += A * (R * ir) * sa * cang;                                 // F_z = -st sz Az
    }
    Px = -Ar * ct - At * sn;
    Py = -Ar * sn + At * ct;
    Pz = -Az;
}

// ---- collision ------------------------------------------------------------------------------
template <class R>
struct Macro { R rho, ux, uy, uz; };

// The moments a collision needs, from v = f - w: drho = sum f - 1, j = sum c f and the raw
// second moments m4..m8 of Eq. (Mmatrix) (xy, xz, yz, x^2 - y^2, x^2 - z^2; the weights
// contribute nothing to them).  Every sum is formed from the z-triplets of the nine
// (cx, cy) columns of the lattice: P = f(+z) + f(-z), S = P + f(0), D = f(+z) - f(-z),
// which roughly halves the additions of summing each moment over its populations.
template <class R>
struct MomentSums { R drho, jx, jy, jz, m4, m5, m6, m7, m8; };

// F32 (the storage): m6 is summed column by column, as collide_f32's results are pinned.
template <class R, bool F32 = false>
__device__ __forceinline__ MomentSums<R> moment_sums(const R (&v)[Q]) {
    R P[3][3], S[3][3], D[3][3];
    sfor<0, 9>([&](auto kc) {                       // column (cx, cy) = (a - 1, b - 1)
        constexpr int k = decltype(kc)::value, a = k % 3, b = k / 3;
        constexpr int ip = dir_of(a - 1, b - 1, 1), im = dir_of(a - 1, b - 1, -1), i0 = dir_of(a - 1, b - 1, 0);
        P[a][b] = add_(v[ip], v[im]);
        S[a][b] = add_(P[a][b], v[i0]);
        D[a][b] = sub_(v[ip], v[im]);
    });
    MomentSums<R> m;
    R Sa[3], Da[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Sa[k] = add_(add_(S[k][0], S[k][1]), S[k][2]);     // column sums at cx = k - 1
        Da[k] = add_(add_(D[k][0], D[k][1]), D[k][2]);
    }
    const R Sb0 = add_(add_(S[0][0], S[1][0]), S[2][0]);   // at cy = -1, +1
    const R Sb2 = add_(add_(S[0][2], S[1][2]), S[2][2]);
    m.drho = add_(add_(Sa[0], Sa[1]), Sa[2]);
    m.jx = sub_(Sa[2], Sa[0]);
    m.jy = sub_(Sb2, Sb0);
    m.jz = add_(add_(Da[0], Da[1]), Da[2]);
    m.m4 = sub_(sub_(S[2][2], S[2][0]), sub_(S[0][2], S[0][0]));
    m.m5 = sub_(Da[2], Da[0]);
    if constexpr (F32) m.m6 = add_(add_(sub_(D[0][2], D[0][0]), sub_(D[1][2], D[1][0])), sub_(D[2][2], D[2][0]));
    else m.m6 = sub_(add_(add_(D[0][2], D[1][2]), D[2][2]), add_(add_(D[0][0], D[1][0]), D[2][0]));
    m.m7 = sub_(add_(S[0][1], S[2][1]), add_(S[1][0], S[1][2]));
    // x^2 - z^2: +1 on the cz = 0 populations of the cx != 0 columns, -1 on the cz != 0
    // populations of the cx = 0 columns
    constexpr int a0 = dir_of(-1, -1, 0), a1 = dir_of(-1, 0, 0), a2 = dir_of(-1, 1, 0);
    constexpr int b0 = dir_of(1, -1, 0), b1 = dir_of(1, 0, 0), b2 = dir_of(1, 1, 0);
    const R f0x = add_(add_(add_(v[a0], v[b0]), add_(v[a1], v[b1])), add_(v[a2], v[b2]));
    m.m8 = sub_(f0x, add_(add_(P[1][0], P[1][1]), P[1][2]));
    return m;
}

// rho and u = sum c f / rho + g / 2 from the sums (bare momentum j, hg = g / 2).  SCALED: the
// sums are in units of inv = 2^-s (the scaled half format; powers of two, exact).
// LEAN takes u = j (1 / rho) + g / 2: the default model in every storage.  The ablation models
// and general rates take u = j + (g / 2 - j (rho - 1) / rho): the bracket is small, so u is
// rounded once.
template <class R, bool SCALED = false, bool LEAN = false>
__device__ __forceinline__ Macro<R> macro_from_sums(const MomentSums<R> &s, R hgx, R hgy, R hgz,
                                                    typename scalar_of<R>::type inv = 1) {
    Macro<R> m;
    R jx = s.jx, jy = s.jy, jz = s.jz;
    if constexpr (LEAN) {
        if constexpr (SCALED) m.rho = fma_(s.drho, lit<R>(inv), lit<R>(1));
        else m.rho = add_(s.drho, lit<R>(1));
        R ir = recip_(m.rho);
        if constexpr (SCALED) ir = mul_(ir, lit<R>(inv));
        m.ux = fma_(jx, ir, hgx);
        m.uy = fma_(jy, ir, hgy);
        m.uz = fma_(jz, ir, hgz);
        return m;
    }
    if constexpr (SCALED) {
        m.rho = fma_(s.drho, lit<R>(inv), lit<R>(1));
        jx = mul_(jx, lit<R>(inv));
        jy = mul_(jy, lit<R>(inv));
        jz = mul_(jz, lit<R>(inv));
    } else {
        m.rho = add_(s.drho, lit<R>(1));
    }
    const R nq = mul_(sub_(lit<R>(1), m.rho), recip_(m.rho));
    m.ux = add_(jx, fma_(jx, nq, hgx));
    m.uy = add_(jy, fma_(jy, nq, hgy));
    m.uz = add_(jz, fma_(jz, nq, hgz));
    return m;
}

template <class R>
__device__ __forceinline__ Macro<R> macroscopic(const R (&v)[Q], R gx, R gy, R gz) {
    return macro_from_sums<R, false, true>(moment_sums<R>(v), mul_(lit<R>(0.5f), gx), mul_(lit<R>(0.5f), gy), mul_(lit<R>(0.5f), gz));
}

// One-axis factors of the product-form equilibrium (see the file header):
// dl[c+1] = psi_hat(c,u) - 1, hd[c+1] = (g/2) d psi_hat / du.
template <class R>
__device__ __forceinline__ void axis_factors(R u, R g, R (&dl)[3], R (&hd)[3]) {
    const R u2 = u * u;
    dl[1] = R(-1.5) * u2;
    dl[0] = R(3) * u2 - R(3) * u;
    dl[2] = R(3) * u2 + R(3) * u;
    const R hg = R(0.5) * g;
    hd[1] = hg * (R(-3) * u);
    hd[0] = hg * (R(6) * u - R(3));
    hd[2] = hg * (R(6) * u + R(3));
}

// Collision models: bit 0 selects the relaxation matrix (0: Lambda of Eq. (lambda);
// 1: Lambda = omega I, the single-relaxation-time operator of Eq. (srt) with the forcing
// term of Eq. (collision)), bit 1 the equilibrium (0: Eq. (BoltzmannEquilibriumDistribution);
// 1: its second-order truncation, the "LBM-O(2)" of Sec. III.B, with the forcing
// populations g . grad_u f^eq, which are Guo et al.'s (2002) for that equilibrium).
enum { MODEL_MRT_H6 = 0, MODEL_BGK = 1, MODEL_O2 = 2, MODEL_RATES = 4 };

// acc + e x for a lattice component e in {-1, 0, 1}; starting from -0 the sum is exact.
template <int E, class R> __device__ __forceinline__ R cterm(R acc, R x) {
    if constexpr (E == 1) return acc + x;
    else if constexpr (E == -1) return acc - x;
    else return acc;
}

// Post-collision populations of the default model (FP64 and 16-bit storage; F32: collide_f32) and
// of the BGK and second-order models, from the moment sums of a cell (R float,
// double) or of a pair of cells (R pf2): emit(i, f*_i - w_i) for every i, row of columns
// (c_y) by row.  SCALED (the scaled half format): sums and outputs are in storage
// units, (f - w) sc with sc = 1 / inv a power of two; the shear moments stay in those units
// and sc enters the density constants, which is exact.
//
//   f*_i - w_i = w_i drho + w_i rho X_i + (shear term), X_i = f^eq / (w rho) - 1 +
//   (1/2) g . grad_u (f^eq / (w rho)).
//
// With the one-axis factors p = psi_hat, d = p - 1, h = (g/2) psi_hat', per in-plane column
// D = px py - 1 = dx + dy px and G = D + hx py + hy px, X = G + hz (1 + D) + dz (1 + G): the
// force meets dz only in the last sum, whose rounding differs from column to column (added to
// dz once for all columns, its rounding adds up over them and the mean flow drifts: the error
// of u after 100 steps doubles).  The shear moments use the bare momentum j and p = j +
// rho g / 2: m_k - m_k^eq + R_k / 2 collapses to m4 - j_x u_y + (g_y / 2) p_x and its like.
// About 290 FP32 operations per cell (330 with rho u u products and separate weights); emitting
// row by row keeps the live set small.
// ACT: the outputs are multiplied by act (1, or 0 for the padding half of a pair, which must
// stay zero) through the four factors they all carry.
// LEAN (see macro_from_sums): X = G (1 + dz) + hz D + (dz + hz), 15 operations fewer.
//
// MODEL_BGK: f* = f + omega (f^eq - f) + (2 - omega) F/2 = f + omega (w drho + w rho X - (f - w))
// with h scaled by (2 - omega) / omega in X; the populations f - w are read from fin.  (Folding
// omega into the weights saves an operation per population and rounds the momentum of all
// of them alike once more: 1.05e-5 instead of 5e-6 off after 1,000 laminar steps.)
// MODEL_O2: X = 9/2 (c.u)(c.w) + 3/2 (c.u + c.w) - 3/2 u.w with w = u + g (that factor times g
// for the BGK), evaluated for c and -c together: even part plus and minus odd part.
template <class R, bool SCALED, bool ACT, bool LEAN, int MODEL = 0, class Emit>
__device__ __forceinline__ Macro<R> collide_mrt(const MomentSums<R> &ms, R gx, R gy, R gz,
                                                typename scalar_of<R>::type omega, typename scalar_of<R>::type inv,
                                                typename scalar_of<R>::type sc, R *s_out, Emit &&emit,
                                                R act = lit<R>(1), const R *fin = nullptr) {
    using S = typename scalar_of<R>::type;
    constexpr bool bgk = (MODEL & MODEL_BGK) != 0, o2 = (MODEL & MODEL_O2) != 0;
    const R hgx = mul_(lit<R>(0.5f), gx), hgy = mul_(lit<R>(0.5f), gy), hgz = mul_(lit<R>(0.5f), gz);
    const Macro<R> mm = macro_from_sums<R, SCALED, LEAN>(ms, hgx, hgy, hgz, inv);
    const R rho = mm.rho;
    // non-equilibrium shear moments s4..s8 (p = j + rho g / 2, in the units of the sums)
    const R rs = SCALED ? mul_(rho, lit<R>(sc)) : rho;
    const R px_ = fma_(rs, hgx, ms.jx), py_ = fma_(rs, hgy, ms.jy), pz_ = fma_(rs, hgz, ms.jz);
    const R njx = neg_(ms.jx), njy = neg_(ms.jy);
    const R s4 = fma_(njx, mm.uy, fma_(hgy, px_, ms.m4));
    const R s5 = fma_(njx, mm.uz, fma_(hgz, px_, ms.m5));
    const R s6 = fma_(njy, mm.uz, fma_(hgz, py_, ms.m6));
    const R tx = fma_(njx, mm.ux, mul_(hgx, px_));            // -rho (u_x^2 - g_x u_x)
    const R ty = fma_(njy, mm.uy, mul_(hgy, py_));
    const R tz = fma_(neg_(ms.jz), mm.uz, mul_(hgz, pz_));
    const R s7 = sub_(add_(ms.m7, tx), ty);
    const R s8 = sub_(add_(ms.m8, tx), tz);
    if (s_out) {
        s_out[0] = s4; s_out[1] = s5; s_out[2] = s6; s_out[3] = s7; s_out[4] = s8;
    }
    // (1 - omega) C_k s_k on the populations with the matching velocity products
    const S om1 = S(1) - omega;
    R om6 = lit<R>(om1 * S(1.0 / 6.0)), om4 = lit<R>(om1 * S(0.25)), rho_o = rho, drho_o = ms.drho;
    if constexpr (ACT) {
        om6 = mul_(om6, act);
        om4 = mul_(om4, act);
        rho_o = mul_(rho_o, act);
        drho_o = mul_(drho_o, act);
    }
    R s12 = lit<R>(0), s34 = s12, s56 = s12, q4 = s12, q5 = s12, q6 = s12;
    R kx = hgx, ky = hgy, kz = hgz;             // half the force that enters X
    if constexpr (bgk) {
        const R kap = lit<R>((S(2) - omega) * recip_(omega));
        kx = mul_(kap, hgx);
        ky = mul_(kap, hgy);
        kz = mul_(kap, hgz);
    } else {
        const R b7 = mul_(om6, s7), b8 = mul_(om6, s8);
        s12 = fma_(om6, s7, b8);
        s34 = fma_(lit<R>(-2), b7, b8);
        s56 = fma_(lit<R>(-2), b8, b7);
        q4 = mul_(om4, s4);
        q5 = mul_(om4, s5);
        q6 = mul_(om4, s6);
    }
    // w rho and w drho (plus the shear term of the population) per weight shell
    const S f = SCALED ? sc : S(1);
    const R wr0 = mul_(lit<R>(S(w_of(0)) * f), rho_o), wr1 = mul_(lit<R>(S(w_of(1)) * f), rho_o);
    const R wr2 = mul_(lit<R>(S(w_of(7)) * f), rho_o), wr3 = mul_(lit<R>(S(w_of(19)) * f), rho_o);
    const R w1 = lit<R>(S(w_of(1))), w2 = lit<R>(S(w_of(7)));
    const R wd0 = mul_(lit<R>(S(w_of(0))), drho_o), wd3 = mul_(lit<R>(S(w_of(19))), drho_o);
    const R c12 = fma_(w1, drho_o, s12), c34 = fma_(w1, drho_o, s34), c56 = fma_(w1, drho_o, s56);
    const R c4p = fma_(w2, drho_o, q4), c4m = fma_(w2, drho_o, neg_(q4)), c5p = fma_(w2, drho_o, q5);
    const R c5m = fma_(w2, drho_o, neg_(q5)), c6p = fma_(w2, drho_o, q6), c6m = fma_(w2, drho_o, neg_(q6));
    auto put = [&](auto ic, R X) {
        constexpr int i = decltype(ic)::value;
        R wr, wd;
        if constexpr (i == 0) { wr = wr0; wd = wd0; }
        else if constexpr (i <= 6) {
            wr = wr1;
            wd = (i <= 2) ? c12 : ((i <= 4) ? c34 : c56);
        } else if constexpr (i <= 18) {
            wr = wr2;
            if constexpr (i == 7 || i == 10) wd = c4p;
            else if constexpr (i == 8 || i == 9) wd = c4m;
            else if constexpr (i == 11 || i == 14) wd = c5p;
            else if constexpr (i == 12 || i == 13) wd = c5m;
            else if constexpr (i == 15 || i == 18) wd = c6p;
            else wd = c6m;
        } else { wr = wr3; wd = wd3; }
        if constexpr (bgk) emit(ic, fma_(lit<R>(omega), sub_(fma_(wr, X, wd), fin[i]), fin[i]));
        else emit(ic, fma_(wr, X, wd));
    };
    if constexpr (o2) {
        const R wx = fma_(lit<R>(2), kx, mm.ux), wy = fma_(lit<R>(2), ky, mm.uy), wz = fma_(lit<R>(2), kz, mm.uz);
        const R ne0 = mul_(lit<R>(-1.5f), fma_(mm.ux, wx, fma_(mm.uy, wy, mul_(mm.uz, wz))));
        put(std::integral_constant<int, 0>{}, ne0);
        sfor<1, Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value, ib = opp_of(i);
            if constexpr (i < ib) {
                auto dot = [](R x, R y, R z) {
                    constexpr int ex = cx_of(i), ey = cy_of(i), ez = cz_of(i);
                    auto term = [](auto e, R acc, R q) {
                        constexpr int k = decltype(e)::value;
                        if constexpr (k == 1) return add_(acc, q);
                        else if constexpr (k == -1) return sub_(acc, q);
                        else return acc;
                    };
                    using std::integral_constant;
                    if constexpr (ex != 0) {
                        const R t = ex > 0 ? x : neg_(x);
                        return term(integral_constant<int, ez>{}, term(integral_constant<int, ey>{}, t, y), z);
                    } else if constexpr (ey != 0) {
                        return term(integral_constant<int, ez>{}, ey > 0 ? y : neg_(y), z);
                    } else {
                        return ez > 0 ? z : neg_(z);
                    }
                };
                const R cu = dot(mm.ux, mm.uy, mm.uz), cw = dot(wx, wy, wz);
                const R even = fma_(mul_(lit<R>(4.5f), cu), cw, ne0), odd = add_(cu, cw);
                put(ic, fma_(lit<R>(1.5f), odd, even));
                put(std::integral_constant<int, ib>{}, fma_(lit<R>(-1.5f), odd, even));
            }
        });
        return mm;
    }
    // one-axis factors at c = -1, 0, +1: d, h and p = 1 + d (those of x row by row).  No sum
    // takes a product that is rounded by itself: the compiler fuses those on pairs and not on
    // single cells, and the two would differ in the last bit.
    auto axis = [](auto cc, R u, R hg, R &d, R &h, R &p) {
        constexpr int c = decltype(cc)::value;
        const R u2 = mul_(u, u), t = mul_(lit<R>(3), u), h3 = mul_(lit<R>(3), hg), w = mul_(h3, u);
        if constexpr (c == 1) {
            d = mul_(lit<R>(-1.5f), u2);
            h = neg_(w);
            p = fma_(lit<R>(-1.5f), u2, lit<R>(1));
        } else {
            d = fma_(lit<R>(3), u2, c == 0 ? neg_(t) : t);
            h = fma_(lit<R>(2), w, c == 0 ? neg_(h3) : h3);
            p = add_(d, lit<R>(1));
        }
    };
    R dy[3], hy[3], py[3], dz[3], hz[3], pz[3], ez[3];
    sfor<0, 3>([&](auto cc) {
        constexpr int c = decltype(cc)::value;
        axis(cc, mm.uy, ky, dy[c], hy[c], py[c]);
        axis(cc, mm.uz, kz, dz[c], hz[c], pz[c]);
        if constexpr (c == 1) ez[c] = fma_(lit<R>(-1.5f), mul_(mm.uz, mm.uz), hz[c]);
        else ez[c] = add_(dz[c], hz[c]);
    });
    sfor<0, 3>([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        R dx, hx, px;
        axis(ac, mm.ux, kx, dx, hx, px);
        sfor<0, 3>([&](auto bc) {
            constexpr int b = decltype(bc)::value;
            const R D = fma_(dy[b], px, dx);
            const R G = fma_(hx, py[b], fma_(hy[b], px, D));
            const R A = add_(D, lit<R>(1)), H = add_(G, lit<R>(1));
            sfor<0, 3>([&](auto cc) {
                constexpr int c = decltype(cc)::value, i = dir_of(a - 1, b - 1, c - 1);
                R X;
                if constexpr (LEAN) X = fma_(G, pz[c], fma_(hz[c], D, ez[c]));
                else X = fma_(dz[c], H, fma_(hz[c], A, G));
                put(std::integral_constant<int, i>{}, X);
            });
        });
    });
    return mm;
}

// The default model in F32 storage, for one cell (R float) or a pair (R pf2): emit as in
// collide_mrt, the same closed form in the order of operations to which the results of F32 runs
// are pinned, bit for bit: a long run adds up what each step rounds (2,000 steps of a decaying
// flow: 5e-5 between two orders), so another order is another result.
//   X = G + hz A + dz H with G = Dxy + Fxy, A = 1 + Dxy, H = A + Fxy per column, Dxy = dx + dy +
//   dx dy, Fxy = hx (1 + dy) + hy (1 + dx); f* - w = w rho X + (w drho + shear term).
// 330 operations per cell, 165 issue slots on pairs.
template <class R, bool ACT, class Emit>
__device__ __forceinline__ Macro<R> collide_f32(const MomentSums<R> &ms, R gx, R gy, R gz, float omega, R *s_out,
                                                Emit &&emit, R act = lit<R>(1)) {
    const R hgx = mul_(lit<R>(0.5f), gx), hgy = mul_(lit<R>(0.5f), gy), hgz = mul_(lit<R>(0.5f), gz);
    const Macro<R> mm = macro_from_sums<R, false, true>(ms, hgx, hgy, hgz);
    const R rho = mm.rho, ux = mm.ux, uy = mm.uy, uz = mm.uz;
    // s_k = m_k - m_k^eq + R_k / 2, k = 4..8
    const R ux2 = mul_(ux, ux), uy2 = mul_(uy, uy), uz2 = mul_(uz, uz);
    const R hr = mul_(lit<R>(0.5f), rho), nrho = neg_(rho), nrx = neg_(mul_(rho, ux)), nry = neg_(mul_(rho, uy));
    const R gxux = mul_(gx, ux);
    const R s4 = fma_(hr, fma_(gy, ux, mul_(gx, uy)), fma_(nrx, uy, ms.m4));
    const R s5 = fma_(hr, fma_(gz, ux, mul_(gx, uz)), fma_(nrx, uz, ms.m5));
    const R s6 = fma_(hr, fma_(gz, uy, mul_(gy, uz)), fma_(nry, uz, ms.m6));
    const R s7 = fma_(rho, fma_(neg_(gy), uy, gxux), fma_(nrho, sub_(ux2, uy2), ms.m7));
    const R s8 = fma_(rho, fma_(neg_(gz), uz, gxux), fma_(nrho, sub_(ux2, uz2), ms.m8));
    if (s_out) {
        s_out[0] = s4; s_out[1] = s5; s_out[2] = s6; s_out[3] = s7; s_out[4] = s8;
    }
    R om1 = lit<R>(1.f - omega), rho_o = rho, drho_o = ms.drho;
    if constexpr (ACT) {
        om1 = mul_(om1, act);
        rho_o = mul_(rho_o, act);
        drho_o = mul_(drho_o, act);
    }
    const R a4 = mul_(om1, s4), a5 = mul_(om1, s5), a6 = mul_(om1, s6), a7 = mul_(om1, s7), a8 = mul_(om1, s8);
    const R six = lit<R>(float(1.0 / 6.0)), third = lit<R>(float(1.0 / 3.0));
    const R w0 = lit<R>(float(w_of(0))), w1 = lit<R>(float(w_of(1))), w2 = lit<R>(float(w_of(7))), w3 = lit<R>(float(w_of(19)));
    const R c12 = fma_(w1, drho_o, mul_(sum_(a7, a8), six));
    const R c34 = fma_(w1, drho_o, fma_(a8, six, neg_(mul_(a7, third))));
    const R c56 = fma_(w1, drho_o, fma_(a7, six, neg_(mul_(a8, third))));
    const R wd2 = mul_(w2, drho_o), wd3 = mul_(w3, drho_o), q = lit<R>(0.25f), nq = lit<R>(-0.25f);
    const R wr0 = mul_(w0, rho_o), wr1 = mul_(w1, rho_o), wr2 = mul_(w2, rho_o), wr3 = mul_(w3, rho_o);
    // one-axis factors at c = -1, 0, +1: d = psi_hat - 1, h = (g / 2) psi_hat'
    auto axis = [](auto cc, R u, R u2, R hg, R &d, R &h) {
        constexpr int c = decltype(cc)::value;
        if constexpr (c == 1) {
            d = mul_(lit<R>(-1.5f), u2);
            h = mul_(hg, mul_(lit<R>(-3.f), u));
        } else {
            const R t = mul_(lit<R>(c == 0 ? -3.f : 3.f), u);
            d = fma_(lit<R>(3.f), u2, t);
            h = mul_(hg, fma_(lit<R>(6.f), u, lit<R>(c == 0 ? -3.f : 3.f)));
        }
    };
    R dy[3], hy[3], oy[3], dz[3], hz[3];
    sfor<0, 3>([&](auto cc) {
        constexpr int c = decltype(cc)::value;
        axis(cc, uy, uy2, hgy, dy[c], hy[c]);
        axis(cc, uz, uz2, hgz, dz[c], hz[c]);
        oy[c] = sum_(dy[c], lit<R>(1));
    });
    sfor<0, 3>([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        R dx, hx;
        axis(ac, ux, ux2, hgx, dx, hx);
        const R ox = sum_(dx, lit<R>(1));
        sfor<0, 3>([&](auto bc) {
            constexpr int b = decltype(bc)::value;
            const R D = fma_(dx, dy[b], sum_(dx, dy[b])), F = fma_(hx, oy[b], mul_(hy[b], ox));
            const R A = add_(D, lit<R>(1)), G = add_(D, F), H = add_(A, F);
            sfor<0, 3>([&](auto cc) {
                constexpr int c = decltype(cc)::value, i = dir_of(a - 1, b - 1, c - 1);
                using I = std::integral_constant<int, i>;
                const R X = fma_(dz[c], H, fma_(hz[c], A, G));
                if constexpr (i == 0) emit(I{}, fma_(w0, drho_o, mul_(wr0, X)));
                else if constexpr (i <= 6) emit(I{}, fma_(wr1, X, i <= 2 ? c12 : i <= 4 ? c34 : c56));
                else if constexpr (i <= 18) {
                    constexpr int k = (i - 7) / 4, e = (i - 7) % 4;          // shear moment 4 + k, sign + - - +
                    emit(I{}, fma_(wr2, X, fma_(e == 0 || e == 3 ? q : nq, k == 0 ? a4 : k == 1 ? a5 : a6, wd2)));
                } else emit(I{}, fma_(wr3, X, wd3));
            });
        });
    });
    return mm;
}

// In-place collision of one fluid cell; v holds f - w on entry and f* - w on exit.
// With s_out, the five non-equilibrium shear moments s_k = m_k - m_k^eq + R_k / 2
// (k = 4..8) are returned as well (the adjoint stores them).
//
// Every model has the form f* = f^eq + F/2 + (1 - omega) N with F = g . grad_u f^eq:
// for the MRT, N = sum_{k=4..8} C_k s_k (the other moments relax with rate 1), and s_k
// is the same for both equilibria since they share their second moments and those of F;
// for the BGK, N = f - f^eq + F/2.  MODEL_RATES takes a general diagonal Lambda:
// f* = f^eq + F/2 + (M^T)^{-1} (1 - Lambda) M^T n with n = f - f^eq + F/2, whose moments
// 0..3 vanish (lam1[k - 4] = 1 - lambda_k).  SCALED (default model only): v is in storage units,
// see collide_mrt.
template <class R, int MODEL = MODEL_MRT_H6, bool SCALED = false, bool LEAN = sizeof(R) == 8>
__device__ __forceinline__ Macro<R> collide(R (&v)[Q], R gx, R gy, R gz, R omega, R *s_out = nullptr,
                                            const R *lam1 = nullptr, R inv = R(1), R sc = R(1)) {
    static_assert(!SCALED || MODEL == MODEL_MRT_H6, "scaled units serve the default model only");
    constexpr bool F32 = MODEL == MODEL_MRT_H6 && !LEAN;
    const MomentSums<R> ms = moment_sums<R, F32>(v);
    if constexpr (F32) {
        return collide_f32<R, false>(ms, gx, gy, gz, omega, s_out, [&](auto ic, R f) { v[decltype(ic)::value] = f; });
    } else if constexpr (!(MODEL & MODEL_RATES)) {
        return collide_mrt<R, SCALED, false, LEAN, MODEL>(ms, gx, gy, gz, omega, inv, sc, s_out,
                                                          [&](auto ic, R f) { v[decltype(ic)::value] = f; }, R(1), v);
    } else {
        constexpr bool o2 = (MODEL & MODEL_O2) != 0;
        const Macro<R> mm = macro_from_sums<R>(ms, R(0.5) * gx, R(0.5) * gy, R(0.5) * gz);
        const R rho = mm.rho, ux = mm.ux, uy = mm.uy, uz = mm.uz, drho = ms.drho;
        R mk[23];                 // moments 4..26 of n = f - f^eq + F/2
#pragma unroll
        for (int k = 0; k < 23; ++k) mk[k] = 0;
        // v_i becomes f^eq + F/2, from the equilibrium part pm1 = f^eq / (w rho) - 1 and
        // frc = (1/2) g . grad_u (f^eq / (w rho))
        auto emit = [&](auto ic, R pm1, R frc) {
            constexpr int i = decltype(ic)::value;
            const R eq = R(w_of(i)) * (drho + rho * pm1), fh = R(w_of(i)) * rho * frc;
            const R ni = v[i] - eq + fh;
            sfor<4, Q>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr int cik = mt_coef(k, i);
                if constexpr (cik != 0) mk[k - 4] += R(cik) * ni;
            });
            v[i] = eq + fh;
        };
        if constexpr (!o2) {
            R dx[3], hx[3], dy[3], hy[3], dz[3], hz[3];
            axis_factors<R>(ux, gx, dx, hx);
            axis_factors<R>(uy, gy, dy, hy);
            axis_factors<R>(uz, gz, dz, hz);
            // per (cx, cy) pair: Dxy = psi_x psi_y - 1 and the x/y force part
            R Dxy[3][3], Fxy[3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    Dxy[a][b] = dx[a] + dy[b] + dx[a] * dy[b];
                    Fxy[a][b] = hx[a] * (R(1) + dy[b]) + hy[b] * (R(1) + dx[a]);
                }
            sfor<0, Q>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                constexpr int a = cx_of(i) + 1, b = cy_of(i) + 1, c = cz_of(i) + 1;
                const R dxy = Dxy[a][b];
                const R axy = R(1) + dxy;
                const R pm1 = dxy + dz[c] * axy;                       // psi_x psi_y psi_z - 1
                const R frc = Fxy[a][b] * (R(1) + dz[c]) + hz[c] * axy; // (1/2) g . grad psi
                emit(ic, pm1, frc);
            });
        } else {
            // second-order equilibrium: f^eq / (w rho) - 1 = 3 c.u + 9/2 (c.u)^2 - 3/2 u.u and
            // (1/2) g . grad_u of it = 3/2 (c.g - u.g) + 9/2 (c.u)(c.g)
            const R uu = ux * ux + uy * uy + uz * uz, ug = ux * gx + uy * gy + uz * gz;
            sfor<0, Q>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                constexpr int ex = cx_of(i), ey = cy_of(i), ez = cz_of(i);
                const R cu = cterm<ez>(cterm<ey>(cterm<ex>(R(-0.0), ux), uy), uz);
                const R cg = cterm<ez>(cterm<ey>(cterm<ex>(R(-0.0), gx), gy), gz);
                const R pm1 = R(3) * cu + R(4.5) * cu * cu - R(1.5) * uu;
                const R frc = R(1.5) * (cg - ug) + R(4.5) * cu * cg;
                emit(ic, pm1, frc);
            });
        }
#pragma unroll
        for (int k = 0; k < 23; ++k) mk[k] *= lam1[k];
        sfor<0, Q>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            R acc = v[i];
            sfor<4, Q>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr double aik = kMtInv.a[i][k];
                if constexpr (aik != 0.0) acc += R(aik) * mk[k - 4];
            });
            v[i] = acc;
        });
        return mm;
    }
}

}  // namespace lbm

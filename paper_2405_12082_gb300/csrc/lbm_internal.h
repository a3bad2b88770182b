// lbm_internal.h -- host-side interface between the C ABI (lbm_api.cu) and the
// per-precision kernel translation units (lbm_f64.cu, lbm_f32.cu, ...).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_device.cuh"

namespace lbm {

// What else a step does: EX_STATS adds u_z^k of the pre-collision state to the FP64 sums,
// EX_MOMENTS stores the adjoint's moments.
enum { EX_NONE = 0, EX_STATS = 1, EX_MOMENTS = 2 };

// FP64 sums of u_z^k, k = 1..4, of one cell (stride between the four sums); single roundings,
// so every kernel adds the same bits.
__device__ __forceinline__ void add_stats(double *s, int64_t stride, double uz) {
    const double uz2 = __dmul_rn(uz, uz);
    s[0] = __dadd_rn(s[0], uz);
    s[stride] = __dadd_rn(s[stride], uz2);
    s[2 * stride] = __fma_rn(uz2, uz, s[2 * stride]);
    s[3 * stride] = __fma_rn(uz2, uz2, s[3 * stride]);
}

// Kernel parameters of the pair kernels (lbm_pair.cuh): a single pipe carries its member in
// the parameters, an ensemble its block table.
struct PairMember {
    const uint32_t *pairinfo;
    const int4 *cellinfo;
    const void *ftabc, *ztab, *dtab, *gz_field;
    int64_t off, doff, scells, t_end;
    int32_t nx, ny, nz, Ps, trig;
    uint32_t ps_mul, ps_shr;
    float gf[3], omegaf;
};
struct PairArgsBase {
    void *pops;
    int64_t stride;
    const StepTime *times;
    int64_t t;
    double *stats;
    void *moments;           // EX_MOMENTS: [9][scells]
    int64_t dstride;
    int32_t tidx;
    float f16_scale, f16_inv;
    uint32_t zero;           // 0 (see k_odd2)
};
struct PairArgsOne : PairArgsBase {
    static constexpr bool kOne = true;
    float stf[1];
    uint32_t nb_plane, nb_mul, nb_shr;
    uint32_t own[27], pull[27];
    PairMember one;
};
struct PairArgsMany : PairArgsBase {
    static constexpr bool kOne = false;
    int32_t n_members;
    float stf[LBM_MAX_MEMBERS];
    int32_t block0[LBM_MAX_MEMBERS + 1];
    uint32_t nb_plane[LBM_MAX_MEMBERS], nb_mul[LBM_MAX_MEMBERS], nb_shr[LBM_MAX_MEMBERS];
    uint32_t own[27], pull[27];              // pull without the plane offset
    PairMember many[LBM_MAX_MEMBERS];
};
// Resident blocks of 128 threads the even pair kernel's registers are cut for (5: 96 registers).
// R = 96 / R = 48 pipe, fraction of the copy bandwidth: F32 5 blocks 0.992 / 0.907 (4: 0.987 /
// 0.897, 6: 0.963 / 0.876).
// The 16-bit formats' two pairs per thread take 128 registers (4 blocks).
constexpr int even_pairs(int precision, int wall) { return precision == LBM_F32 || wall == LBM_BOUZIDI ? 1 : 2; }
constexpr int EVEN2_THREADS = 128;
template <int P, int WALL> constexpr int EVEN2_BLOCKS = even_pairs(P, WALL) == 1 ? 5 : 4;
// Planes the odd pair kernel takes singly (0, nz - 1 and, for odd nz > 2, nz - 2), and its plane
// groups of zc planes (the pairs 1 .. nz - 2) after them.
__host__ __device__ inline int odd_single_planes(int nz) { return nz < 3 ? nz : 2 + (nz & 1); }
__host__ __device__ inline int odd_pair_groups(int nz, int zc) { return nz < 3 ? 0 : ((nz - 2) / 2 * 2 + zc - 1) / zc; }
inline void fill_pair_args(PairArgsBase &o, const StepArgs &a) {
    o.pops = a.pops; o.stride = a.stride; o.times = a.times; o.t = a.t; o.stats = a.stats; o.moments = a.moments; o.dstride = a.dstride;
    o.tidx = a.tidx; o.zero = 0; o.f16_scale = a.f16_scale; o.f16_inv = a.f16_inv;
}
inline void fill_pair_member(PairMember &o, const Member &d) {
    o.pairinfo = d.pairinfo; o.cellinfo = d.cellinfo; o.ftabc = d.ftabc; o.ztab = d.ztab; o.dtab = d.dtab;
    o.gz_field = d.gz_field; o.off = d.off; o.doff = d.doff; o.scells = d.scells; o.t_end = d.t_end;
    o.nx = d.nx; o.ny = d.ny; o.nz = d.nz; o.Ps = d.Ps; o.trig = d.trig; o.ps_mul = d.ps_mul; o.ps_shr = d.ps_shr;
    for (int k = 0; k < 3; ++k) o.gf[k] = d.gf[k];
    o.omegaf = d.omegaf;
}

// Programmatic dependent launch.  A step launched with overlap = true may be brought onto the
// GPU while the step before it drains: it announces its own successor at once, reads its
// (constant) tables and then waits until every block of the step before it has finished and
// its writes are visible.  The one-cell, pair and adjoint kernels have both calls; without the
// launch attribute they do nothing.  The pipelined and the staged kernels (shapes 4, 5, 11, 12) have
// neither: their launchers never set the attribute, with which they would race.
__device__ __forceinline__ void release_next_step() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void await_previous_step() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

inline cudaLaunchConfig_t step_config(int blocks, int threads, bool overlap, cudaLaunchAttribute (&at)[1], cudaStream_t s) {
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cfg;
}
template <class A>
cudaError_t launch_step_kernel(void (*kern)(const A), int blocks, int threads, bool overlap, const A &a, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = step_config(blocks, threads, overlap, at, s);
    return cudaLaunchKernelEx(&cfg, kern, a);
}

constexpr int MODES_MAX_THETA = 4096;        // samples of a ring (lbm_modes)
struct ModesArgs {
    int32_t n_sections, n_rings, n_theta, n_modes;
    double r_over_R[16];
};

// Launch shapes of the step kernel ("variants"): threads per block, the number of
// resident blocks per SM the register budget is cut for, the planes each thread takes
// (zc), whether it is the software-pipelined persistent kernel (shapes 4 and 5, F32
// storage only) and whether it is the persistent kernel whose loads are staged in shared
// memory by bulk copies (shapes 11 and 12, compact pipe layouts, every storage; staged =
// index into STAGED_SHAPES + 1).  FP64 storage has shape 0 (32 x 16) and the staged ones.
// Shapes 6-10 (several planes per thread) run on pairs of cells in the compact pipe layouts
// (lbm_pair.cuh): pt, pb, pz are the threads, resident blocks and planes per thread of their
// odd steps there; zc, threads and min_blocks hold for the dense layouts.
// Odd steps, measured on the R = 96 / R = 48 pipes: 128 threads x 4 blocks (128 registers, no
// spills) 1176 / 131 us in F32 with 2 planes per thread, 1187 / 138 us with 4 (the last wave of
// blocks is longer); 128 x 5 spills and takes 1305 / 150 us, 256 x 2 takes 1211 / 138.  F16S:
// 894 / 101 us with 2 planes, 866 / 104 with 4; BF16 891 / 101 and 866 / 105.  Bouzidi walls in
// F32: 1364 / 151 us with 2 planes, 1293 / 151 with 4 (fewer loads of the link coefficients).
struct StepShape { int threads, min_blocks, zc, pipelined, staged, pt, pb, pz; };
constexpr StepShape STEP_SHAPES[13] = {{256, 4, 1, 0, 0, 0, 0, 0},    {256, 3, 1, 0, 0, 0, 0, 0},   {128, 8, 1, 0, 0, 0, 0, 0},
                                       {512, 2, 1, 0, 0, 0, 0, 0},    {256, 3, 1, 1, 0, 0, 0, 0},   {128, 6, 1, 1, 0, 0, 0, 0},
                                       {128, 8, 2, 0, 0, 256, 2, 2},  {128, 8, 4, 0, 0, 128, 4, 4}, {256, 4, 2, 0, 0, 64, 8, 4},
                                       {128, 7, 2, 0, 0, 128, 4, 2},  {128, 6, 2, 0, 0, 128, 4, 8}, {992, 1, 1, 0, 1, 0, 0, 0},
                                       {512, 1, 1, 0, 2, 0, 0, 0}};
// FP64 steps are bound by the FP64 units of each SM: blocks of one warp spread a small context
// evenly over the SMs.
constexpr StepShape STEP_SHAPE_F64 = {32, 16, 1, 0, 0, 0, 0, 0};
// Where a shape of several planes per thread runs one (see shape_run): shape 2.
constexpr int SINGLE_VARIANT = 2, SINGLE_THREADS = STEP_SHAPES[SINGLE_VARIANT].threads;
constexpr int N_STEP_SHAPES = 13;
// Staged shapes: threads per CTA (one producer warp, the rest consume), pipeline stages
// (tiles in flight per CTA), CTAs per SM and consumer groups (tiles worked on at once).
struct StagedShape { int threads, stages, ctas_per_sm, groups; };
constexpr StagedShape STAGED_SHAPES[2] = {{992, 3, 1, 2}, {512, 3, 1, 1}};
inline int staged_of(int variant) {
    return (variant >= 0 && variant < N_STEP_SHAPES) ? STEP_SHAPES[variant].staged - 1 : -1;
}
inline size_t esize_of_precision(int precision) {
    return precision == LBM_F64 ? 8 : (precision == LBM_F32 ? 4 : 2);
}
// Storage elements per direction segment of staged shape k: the largest multiple of 64
// whose STAGES stages (27 segments + a 16-byte cell-table entry per element each) and
// mbarriers fit the shared memory of one CTA when ctas_per_sm CTAs share an SM (GB300:
// 227 KB per CTA, 228 KB per SM with 1 KB reserved per CTA).
inline int staged_cap(int precision, int k) {
    const StagedShape &sh = STAGED_SHAPES[k];
    const int budget = (sh.ctas_per_sm == 1 ? 232448 : (233472 / sh.ctas_per_sm - 1024)) - 80 * sh.stages - 128;
    const int per = sh.stages * (27 * (int)esize_of_precision(precision) + 16);
    return budget / per / 64 * 64;
}
inline int step_variants(int) { return N_STEP_SHAPES; }
// the fastest shapes in sweeps on GB300 (see STEP_SHAPES; even steps run the same pair kernel
// in shapes 6-10).  Odd steps of the 16-bit formats and of Bouzidi walls: 4 planes per thread
// on large contexts, 2 below about 10 M stored cells, where 4 leave too few waves of blocks
// (F16S: R = 96 pipe, 36 M cells, 866 against 894 us; R = 48 pipe, 3.9 M, 104 against 101 us).
inline int default_variant(int precision, int wall) {
    if (precision == LBM_F64) return 0;
    if (wall == LBM_BOUZIDI) return 7;
    return precision == LBM_F32 ? 6 : 7;
}
inline int default_variant_odd(int precision, int wall, int64_t stored_cells) {
    if (precision == LBM_F64) return 0;
    return (wall == LBM_BOUZIDI || precision != LBM_F32) && stored_cells >= 10000000 ? 7 : 9;
}
// the shape the ablation collision models are compiled for (one plane per thread)
inline int model_variant(int precision) { return precision == LBM_F64 ? 0 : 2; }
// the shape of the adjoint's moment-storing steps: pairs of cells where the context has them
// (shape 9), else 256 x 4 with one plane per thread (two planes measured 2 % slower there)
constexpr int MOM_VARIANT = 0, MOM_VARIANT_PAIRS = 9;
// whether the storage can run the shape at all (a staged shape also needs a compact pipe
// layout whose row groups fit its segments: checked per context)
inline bool step_variant_ok(int precision, int variant) {
    if (variant < 0 || variant >= N_STEP_SHAPES) return false;
    if (STEP_SHAPES[variant].staged) return true;
    if (precision == LBM_F64) return variant == 0;
    return precision == LBM_F32 || !STEP_SHAPES[variant].pipelined;
}
inline int step_threads(int precision, int variant) {
    if (precision == LBM_F64 && !STEP_SHAPES[variant].staged) return STEP_SHAPE_F64.threads;
    return STEP_SHAPES[variant].threads;
}
inline int step_zc(int precision, int variant) { return precision == LBM_F64 ? 1 : STEP_SHAPES[variant].zc; }

// Sets the shared-memory size of the staged step kernels of shape `variant` for every
// parity, wall and statistics setting of storage P (once per process; called before any
// graph capture so that the launches being captured only launch).
template <int P>
cudaError_t prepare_step(int wall, int variant);
// Step of a staged shape (lbm_staged.cuh; compiled in lbm_staged_*.cu).
template <int P>
cudaError_t launch_step_staged(int wall, int parity, bool stats, const StepArgs &a, int variant, cudaStream_t s);

// Every launcher enqueues on `s` and returns the launch status.
// Step kernel over all members: a flat grid of a.nblocks_total blocks of
// step_threads(P, variant) threads.
template <int P>
cudaError_t launch_step(int wall, int parity, bool stats, const StepArgs &a, const Member *hm, int variant,
                        cudaStream_t s);

// Forward step that also stores rho, u, s4..s8 into a.moments (adjoint recompute;
// single half-way pipe, F32 or F64 storage, in shape MOM_VARIANT or MOM_VARIANT_PAIRS).
template <int P>
cudaError_t launch_step_moments(int parity, const StepArgs &a, const Member *hm, cudaStream_t s);

// One backward step of the adjoint (see k_adjoint): blocks of ADJ_THREADS threads, each taking
// ADJ_ZC consecutive planes of one stored position in pairs (FP32) or one plane (FP64).
constexpr int ADJ_THREADS = 128, ADJ_ZC = 2;
struct AdjMember {
    const int4 *cellinfo;
    const void *gz_field;
    int32_t nx, ny, nz, Ps;
    uint32_t n;               // stored cells: the stride of the adjoint and moment fields
    float gf[3], omegaf;
    double g[3], omega;
};
struct AdjArgs {
    const void *lam_next;     // lambda_{t+1}, [27][cells] in the compute type
    void *lam;                // lambda_t (written)
    const void *moments;      // [9][cells] of step t: rho, u_x, u_y, u_z, s4..s8
    double *acc;              // [cells]: dJ/dg_z (accumulated, FP64, dense cells)
    void *acc_seg;            // [stored cells]: dJ/dg_z of the current segment (compute type;
                              // added into acc and cleared after each segment)
    double *blockacc;         // [2][nblocks * warps]: objective and dJ/domega per warp (accumulated)
    int32_t objective;        // LBM_J_UBULK | LBM_J_WSS
    double kappa;             // UBULK: 1 / (T N_fluid)
    double wss;               // WSS: 2 / (T 2 pi R nz)
    float kappa_f, wss_f;     // the same in float
    int32_t nblocks;
    uint32_t nb_plane, nb_mul, nb_shr;       // blocks per plane
    uint32_t zero;            // 0 (see adjoint_cells)
    uint32_t own[27], pull[27];              // element offsets, as in the odd step (see lbm_pair.cuh)
    AdjMember one;
};
template <class S> __device__ __forceinline__ S adj_g(const AdjMember &d, int k) {
    if constexpr (sizeof(S) == 4) return d.gf[k]; else return d.g[k];
}
template <class S> __device__ __forceinline__ S adj_omega(const AdjMember &d) {
    if constexpr (sizeof(S) == 4) return d.omegaf; else return d.omega;
}
template <class S> __device__ __forceinline__ S adj_wss(const AdjArgs &j) {
    if constexpr (sizeof(S) == 4) return j.wss_f; else return j.wss;
}
template <class S> __device__ __forceinline__ S adj_kappa(const AdjArgs &j) {
    if constexpr (sizeof(S) == 4) return j.kappa_f; else return j.kappa;
}
template <int P>
void prepare_adjoint(AdjArgs &j, const Member &d);
template <int P>
cudaError_t launch_adjoint(bool overlap, const AdjArgs &j, cudaStream_t s);
// acc[dense cell] += acc_seg[stored cell]; acc_seg = 0 (member 0 of a, compact layout).
template <int P>
cudaError_t launch_flush_segment(const StepArgs &a, const Member &hm, const AdjArgs &j, cudaStream_t s);
// Deterministic column sums of nv <= 5 double arrays [nv][n] into out[5] (device).
template <int P>
cudaError_t launch_sum_columns(const double *base, int64_t n, int nv, double *partials, int n_partials_max,
                               double *out, cudaStream_t s);

// Per-member kernels: member m of a.members (host copy hm for sizes).
template <int P>
cudaError_t launch_moments(int wall, int parity, const StepArgs &a, const Member &hm, int m,
                           void *rho, void *u, cudaStream_t s);
template <int P>
cudaError_t launch_get_pops(int wall, int parity, const StepArgs &a, const Member &hm, int m,
                            double *f, cudaStream_t s);
template <int P>
cudaError_t launch_set_pops(int wall, int parity, const StepArgs &a, const Member &hm, int m,
                            const double *f, cudaStream_t s);
template <int P>
cudaError_t launch_init(int wall, const StepArgs &a, const Member &hm, int m, int profile, double noise_amp,
                        uint64_t seed, const double *rho, const double *u, cudaStream_t s);
// Block partials (5 doubles per block) then a one-block final pass into out[5] (device).
template <int P>
cudaError_t launch_reduce(int wall, int parity, const StepArgs &a, const Member &hm, int m,
                          double *partials, int n_partials_max, double *out, cudaStream_t s);
template <int P>
cudaError_t launch_modes(int wall, int parity, const StepArgs &a, const Member &hm, int m,
                         const ModesArgs &ma, double *E, cudaStream_t s);

// Trigger-force tables of member m (column factors [3][ny][nx], z factors [2][nz]).
template <int P>
cudaError_t launch_force_tables(const Member *dmembers, const Member &hm, int m, void *ftab, void *ztab,
                                cudaStream_t s);

// Records the reason of a failed call that has no context (reported by
// lbm_last_error(NULL) in the calling thread).
void set_thread_error(const char *msg);

constexpr int REDUCE_BLOCK = 256;
constexpr int REDUCE_MAX_BLOCKS = 1216;   // 8 resident blocks x 152 SMs

}  // namespace lbm

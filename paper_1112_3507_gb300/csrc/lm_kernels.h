// Host-visible kernel interfaces of the solver library (internal).
#pragma once

#include <cuda_runtime.h>

#include "lm_common.cuh"
#include "lm_intfp.cuh"

namespace lm {

// Number of kernels this library has launched (all grids, all streams).
void count_launches(long long n);

// Float64 operator: c~, minus-face conductances per axis, inverse diagonal.
struct Op64 {
    const double* ct;
    const double* gx;
    const double* gy;
    const double* gz;
    const double* dinv;
};
struct Op64Out {
    double* ct;
    double* gx;
    double* gy;
    double* gz;
    double* dinv;
    float* ct32;
    float* rho32;
};

struct PcgArgs {
    Geo g;
    Op64 op;
    const double* f;
    double* x;
    double* r;
    double* p;
    double* q;
    double* part;     // NSLOT * MAX_PARTIALS
    SolveState* st;
    double* hist;     // max_iter + 1
    int max_iter;
};

// One float32 multigrid level (device view).  Faces are formed on the fly
// from rho: g = 2 (1/h^2) / (rho_L + rho_R).
struct Lev32 {
    Geo g;
    float c2x, c2y, c2z;     // 2/h^2 per axis
    const float* ct;
    const float* rho;
};

// What the assembly reports besides the coefficients: the range of rho^{n+1}
// (float64 bit patterns, monotone in the value for positive numbers), a
// positivity/finiteness failure, and a c~ outside float32 range.
struct AsmFlags {
    unsigned long long rho_max;
    unsigned long long rho_min;
    int bad;        // rho, c_s^2, dt or c~ not strictly positive and finite
    int bad32;      // c~ overflows or underflows float32
};

// Everything the assembly of one grid reads and writes.
struct AsmArgs {
    Geo g;
    const double* a_in;      // rho^n (or c~ when raw)
    const double* rho_new;
    const double* cs2;
    double dt;
    int raw;
    double c2x, c2y, c2z;    // 2 / h^2 per axis
    int kx, ky, kz;          // their exponents where they are powers of two (pow2_of)
    Op64Out out;
    AsmFlags* fl;
};
inline AsmArgs asm_args(const Geo& g, const double* a_in, const double* rho_new, const double* cs2, double dt,
                        int raw, const double h[3], const Op64Out& out, AsmFlags* fl) {
    const double c[3] = {2.0 / (h[0] * h[0]), 2.0 / (h[1] * h[1]), 2.0 / (h[2] * h[2])};
    return AsmArgs{g,    a_in, rho_new, cs2, dt, raw, c[0], c[1], c[2], pow2_of(c[0]), pow2_of(c[1]), pow2_of(c[2]),
                   out, fl};
}

// fp64
void launch_assemble(const Geo& g, int G, cudaStream_t s, const double* a_in, const double* rho_new,
                     const double* cs2, double dt, int raw, const double h[3], const Op64Out& out, AsmFlags* fl,
                     int i0 = 0, int i1 = -1);
// x *= scale (float32; scale a power of two, so the scaling is exact)
void launch_scale32(int N, int G, cudaStream_t s, float* x, float scale);
void launch_jacobi_diag(const Geo& g, int G, cudaStream_t s, const Op64& op, double* dinv);
void launch_apply64(const Geo& g, int G, cudaStream_t s, const Op64& op, const double* x, double* y,
                    double* part);
void launch_pcg_init(const PcgArgs& a, int G, cudaStream_t s, int use_x0);
void launch_pcg_restart(const PcgArgs& a, int G, cudaStream_t s, int k);
// the operator-free steps of one Jacobi-PCG iteration, for operators applied
// elsewhere: p = D^-1 r with r.z (after the residual), the x, r update after
// q = A p with its p.q partials (slot 0), and the convergence test with the p update
void launch_pcg_init_p(const PcgArgs& a, int G, cudaStream_t s, int rz_slot, int restart);
void launch_pcg_xr(const PcgArgs& a, int G, cudaStream_t s, int k);
void launch_pcg_p(const PcgArgs& a, int G, cudaStream_t s, int k);
void launch_pcg_iter(const PcgArgs& a, int G, cudaStream_t s, int k);
// iterations k0 .. k1 - 1 (or until done) in one cooperative kernel, for grids
// it fits on a device of nsm SMs; from_part: r.z is in the partials (first
// launch after an init or restart), else in st->scale; bar: two words; looks: of
// a waiting block at a grid barrier before it gives up.  LM_ERR_CUDA: refused,
// nothing has run.
bool pcg_run_fits(int N, int G, int nsm);
int launch_pcg_run(const PcgArgs& a, int G, int nsm, cudaStream_t s, int k0, int k1, int from_part, unsigned* bar,
                   unsigned looks);
void launch_true_residual(const PcgArgs& a, int G, cudaStream_t s);
void launch_ir_residual(const Geo& g, int G, cudaStream_t s, const Op64& op, const double* f, double* x,
                        float* r32, double* part, int zero_x, SolveState* st, int set_fnorm, double* hist_entry,
                        double rscale = 1.0);
void launch_warm_scale(const Geo& g, int G, cudaStream_t s, const Op64& op, const double* f, double* x,
                       double* part);
void launch_ir_correct(int N, int G, cudaStream_t s, double* x, const float* e, double escale = 1.0);
void launch_reduce_rel(double* part, int G, cudaStream_t s, SolveState* st, double* hist_entry);
void launch_reduce_slot(const double* part, int slot, int G, cudaStream_t s, double* out);
void launch_fcg64_iter_a(int N, int G, cudaStream_t s, const float* z, const double* q, double* part, int first,
                         double* p, const SolveState* st);
void launch_fcg64_iter_b(const Geo& g, int G, cudaStream_t s, const Op64& op, double* x, double* r, float* r32,
                         const double* p, double* q, double* part, SolveState* st);
void launch_to32(int N, int G, cudaStream_t s, const double* r, float* r32);
void launch_set_fnorm(const double* part, int slot, int G, cudaStream_t s, SolveState* st);

// fp32 operator and flexible CG (reductions land in red.scal[slot]; slot < 0: none)
void launch_apply32(const Lev32& L, cudaStream_t s, const float* x, float* y, const float* r, const Red& red,
                    int slot_xy, int slot_xr);
void launch_dot32(int N, int G, cudaStream_t s, const float* a, const float* b, const Red& red, int slot,
                  SolveState* fnorm_st);
void launch_axpy32(int N, int G, cudaStream_t s, float alpha, const float* x, const float* y, float* out);
void launch_axpy_ratio32(int N, int G, cudaStream_t s, const double* scal, int num, int den, const float* x,
                         const float* y, float* out);
void launch_fcg_beta_p(int N, int G, cudaStream_t s, const float* z, float* p, const double* scal, int first);
void launch_fcg_update(int N, int G, cudaStream_t s, float* e, float* r, const float* p, const float* q,
                       const Red& red, SolveState* st);

// multigrid
void launch_coarsen(const Lev32& F, const Lev32& C, int hx, int hy, int hz, cudaStream_t s, float* ct_c,
                    float* rho_c);
void launch_rbgs(const Lev32& L, cudaStream_t s, const float* xin, const float* ec, const Lev32* C, int hx, int hy,
                 int hz, const float* f, float* xout, int first, int zero, int prolong);
void launch_rbgs_kz(const Lev32& L, cudaStream_t s, const float* xin, const float* ec, const Lev32* C, int hx,
                    int hy, int hz, const float* f, float* xout, int first, int zero, int prolong, int kz);
void launch_resid_restrict(const Lev32& F, const Lev32& C, int hx, int hy, int hz, cudaStream_t s,
                           const float* x, const float* f, float* fc);
// A whole coarse V-cycle in one launch (lm_coarse.cuh): the levels of a chain
// down to the coarsest, which is solved with its dense inverse or, when it has
// none, by COARSE_SWEEPS sweep pairs.  A level of up to CC_MAX_PAIRS pairs of
// x-neighbours (4096 cells with even rows; CC_PER pairs a thread is what its
// registers hold) is run by one block, a larger one by the blocks of a cluster.
constexpr int COARSE_SWEEPS = 32;                // (red-black, black-red) sweep pairs of an unsolved coarsest level
constexpr int CC_MAXL = 8;
constexpr int CC_THREADS = 512;                  // threads of a block that runs a cycle
constexpr int CC_PER = 4;                        // pairs a thread owns on a chain level, at most
constexpr int CC_MAX_PAIRS = CC_THREADS * CC_PER;
constexpr int CC_PER_SHARED = 2;                 // ... on a level that the blocks of a cluster share
constexpr int CC_CLUSTER = 16;                   // blocks of a cluster (the hardware's most)
constexpr size_t CC_SMEM_MAX = 200 * 1024;       // shared-memory limit of a block
// How a level's Gauss-Seidel values are formed: like the kernels that sweep
// such a level on its own, weights face by face and an approximate division by
// the diagonal (rbgs_tile) or one reciprocal for the two faces of an axis
// (zrow2d_tile); or face by face with the correctly rounded inverse diagonal
// (the levels of an exactly solved chain, see inverse_level).
enum CCArith { CC_FACE, CC_AXIS, CC_INVERSE };
struct CCLevel {
    Lev32 L;
    int hx, hy, hz;                // halvings to the next chain level
    int nr;                        // blocks that share the level (never more than on the level before)
    int arith;                     // CCArith
    int hp, halo;                  // pairs a row; planes of halo each side (0: one block)
    int npair, ncell, off;         // floats of an array by staged pair and by own cell; where the level's arrays lie
    float ix, iy, iun, inr, imean; // 1 / nx, ny, units, nr, children of a cell of the next level
    float4* plan;                  // the level's pairs as cc_plan_pair lays them out (not a solved coarsest level)
};
struct CoarseCycle {
    int nl;                        // levels in the chain
    CCLevel lev[CC_MAXL];
    int inv;                       // shared-memory offset (floats) of the dense inverse
    int parts;                     // threads that share a row of it
    float* x;                      // solution of chain level 0
    const float* f;                // its right-hand side
    const float* ainv;             // dense inverse of the coarsest level, or null
    int nu1, nu2;
};
__host__ __device__ inline int cc_align4(int n) { return (n + 3) & ~3; }
__host__ __device__ inline int cc_pairs(const Geo& g) { return ((g.nx + 1) >> 1) * g.ny * g.nz; }
// A shared level is split into units of the planes that make one plane of the
// next level; block r of nr owns the units from cc_unit0(r) to cc_unit0(r + 1).
__host__ __device__ inline int cc_unit0(int r, int units, int nr) { return r * units / nr; }
__host__ __device__ inline int cc_owner(int unit, int units, int nr) { return ((unit + 1) * nr - 1) / units; }
// The most planes a block owns.
__host__ __device__ inline int cc_own(const CCLevel& v) {
    const int units = v.L.g.nz >> v.hz;
    return ((units + v.nr - 1) / v.nr) << v.hz;
}
// Fills the derived fields of the levels, lays a block's shared memory out
// (per level the two colours of x by staged pair, right-hand side and residual
// by own cell) and returns its bytes.
inline size_t cc_layout(CoarseCycle& cc) {
    size_t o = 0;
    for (int l = 0; l < cc.nl; ++l) {
        CCLevel& v = cc.lev[l];
        const Geo& g = v.L.g;
        v.hp = (g.nx + 1) >> 1;
        v.halo = v.nr > 1 ? 1 : 0;
        const int own = cc_own(v);
        v.npair = cc_align4(v.hp * g.ny * (own + 2 * v.halo));
        v.ncell = cc_align4(g.nx * g.ny * own);
        v.off = (int)o;
        v.ix = 1.f / (float)g.nx;
        v.iy = 1.f / (float)g.ny;
        v.iun = 1.f / (float)(g.nz >> v.hz);
        v.inr = 1.f / (float)v.nr;
        v.imean = 1.f / (float)((1 << v.hx) << v.hy << v.hz);
        o += 2 * (size_t)v.npair + 2 * (size_t)v.ncell;
    }
    cc.inv = (int)o;
    const size_t nc = (size_t)cc.lev[cc.nl - 1].L.g.N;
    if (cc.ainv) o += nc * nc;
    return sizeof(float) * o;
}
constexpr int CC_PLAN = 6;                       // float4 arrays of a level's plan
// forms the plan of cc's levels (cc.x, cc.f unused), or of `count` chains in device memory
void launch_cc_plan(const CoarseCycle& cc, cudaStream_t s);
void launch_cc_plan_many(const CoarseCycle* ccs, int count, cudaStream_t s);
void launch_coarse_cycle(const CoarseCycle& cc, size_t smem, cudaStream_t s);
// raises k_coarse_cycle's shared-memory and cluster-size limits; returns the
// cluster size it can be launched with (1: no cluster)
int coarse_cycle_allow();
void rbgs_row_allow_smem();                      // raises the whole-row sweep's dynamic shared-memory limit
void launch_coarse_inverse(const Lev32& L, cudaStream_t s, float* ainv);
// one grid's coarsest level and where its dense inverse goes
struct CoarseInv {
    Lev32 L;
    float* ainv;
};
// rows (task & 255) of items[task >> 8] for every task: many grids' inverses in one launch
void launch_coarse_inverse_many(const CoarseInv* items, const int* task, int ntask, cudaStream_t s);
// one block per item: each grid's whole inverse (the factorisation done once per grid)
void launch_coarse_inverse_grids(const CoarseInv* items, int count, cudaStream_t s);
void launch_coarse_solve(int n, cudaStream_t s, const float* ainv, const float* f, float* x);

}  // namespace lm

// The coarse V-cycle in one launch (k_coarse_cycle: a thread-block cluster;
// kb_coarse_cycle: one block per grid of a batch): every level from the first
// one small enough down to the coarsest, in shared memory, in place of six
// launches a level and cycle (64 on a coarsest level without a dense inverse).
//
// What bounds it: the serial chain of half-sweeps (ten a level and cycle with
// two and three sweeps, 65 on an unsolved coarsest level), each a few
// shared-memory reads, dependent multiply-adds and a barrier.  So a half-sweep
// does nothing else.  A thread owns pairs of x-neighbours (one red and one
// black cell each) and keeps their face weights, right-hand sides, inverse
// diagonals and neighbour positions in registers for a level's whole
// smoothing; x alone lives in shared memory, one array per colour, indexed by
// pair, so that a half-sweep reads one array at consecutive addresses (no bank
// conflicts) and writes the other.  Weights and positions are formed once per
// hierarchy, by k_cc_plan, in the order the threads load them: formed inside
// the cycle, their code (executed once per level and leg, so always fetched
// anew) took 38 of the 43 us of a 64 x 64 cycle.
//
// One cycle of two and three sweeps, kernels alone in a graph (one launch a
// level, sweep and transfer and one block below 4096 cells -> here): 64 x 64
// 64.7 -> 20.0 us, 128 x 128 103.6 -> 40.6 us, 30 x 18 x 11 without a dense
// inverse 543 -> 36.5 us.  A half-sweep of one block takes 0.13 us; of a
// cluster 0.5 us, of which the barrier (with the release of the halo stores)
// is 0.33 us whatever the cluster's size.
//
// A level of up to CC_MAX_PAIRS pairs is run by the cluster's first block
// alone, with a barrier over the warps that own pairs.  A larger one is split
// into runs of planes (in 2D rows), one a block: a block keeps its planes and a
// halo of one each side, and a thread that updates a boundary pair also stores
// the value into the neighbouring block's halo (distributed shared memory), so
// every read stays local and a half-sweep ends with one hardware cluster
// barrier.  The planes that make one plane of the next level stay together, so
// a block restricts and prolongs from its own memory: restricted right-hand
// sides and corrections are stored into their owner's.
//
// Registers: the 128 that 512 threads leave each hold four pairs of a 2D level,
// but not of a 3D one, nor what a cluster's kernel carries beside its own two.
// By the compiler's count k_coarse_cycle<1, true> spills 148 bytes a thread
// (176 loaded back), <16, false> 390 (704), <16, true> 666 (1456), partly
// inside the half-sweeps; <1, false> and kb_coarse_cycle nothing.  What they
// would take without was not measured.
//
// The arithmetic of a level is that of the kernel that sweeps such a level on
// its own (CCArith), term by term, so a solve's iterates do not depend on
// where the chain starts.
#pragma once

#include <type_traits>

#include "lm_kernels.h"
#include "lm_tiles.cuh"

namespace lm {

// n floats from global to shared memory, asynchronously.
__device__ __forceinline__ void cc_copy(float* dst, const float* src, int n, int tid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if ((n & 3) == 0 && (((uintptr_t)src | d) & 15) == 0) {
        for (int e = tid; e < (n >> 2); e += CC_THREADS)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + 16 * e), "l"(src + 4 * e) : "memory");
    } else {
        for (int e = tid; e < n; e += CC_THREADS)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * e), "l"(src + e) : "memory");
    }
}

// ---- cluster helpers (NR = 1: a plain block, none is called) ----
__device__ __forceinline__ int cc_rank() {
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cc_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of block `rank`'s copy of this block's shared-memory location p
__device__ __forceinline__ unsigned cc_remote(const float* p, int rank) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cc_st_remote(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// e / n for 0 <= e < 2^22 and inv = 1.f / n: the product is off by less than
// half a unit of 1 / n.
__device__ __forceinline__ int cc_div(int e, float inv) { return (int)(((float)e + 0.5f) * inv); }

// A block's share of a level: planes k0 .. k1 - 1, and the level's shared
// arrays (the same offsets in every block).  A pair's position in x0, x1 is
// m + hp (j + ny (k - k0 + halo)); f and res (a residual on the way down, the
// next level's correction on the way up) go by cell of the own planes.
struct CCLev {
    int k0, k1;
    float *x0, *x1, *f, *res;
};
__device__ __forceinline__ int cc_first(const CCLevel& v, int rank) {        // first plane of a block
    return v.nr > 1 ? cc_div(rank * (v.L.g.nz >> v.hz), v.inr) << v.hz : (rank ? v.L.g.nz : 0);
}
__device__ __forceinline__ int cc_block_of(const CCLevel& v, int k) {        // the block that owns plane k
    return v.nr > 1 ? cc_div(((k >> v.hz) + 1) * v.nr - 1, v.iun) : 0;
}
__device__ __forceinline__ CCLev cc_lev(float* sm, const CCLevel& v, int rank) {
    CCLev s;
    s.k0 = cc_first(v, rank);
    s.k1 = cc_first(v, rank + 1);
    s.x0 = sm + v.off;
    s.x1 = s.x0 + v.npair;
    s.f = s.x1 + v.npair;
    s.res = s.f + v.ncell;
    return s;
}

// ---- the plan: per pair of cells (2m, 2m + 1) of a row, by colour (0 red) ------
//
// Six float4 arrays of a level's pairs in row order (q = 0: x and z face
// weights of the red cell, 1: of the black cell, 2: inverse diagonals and
// positions, 3: own cell index and flags, halo copies, c~; 3D: 4 y weights;
// CC_AXIS levels: 4, 5 the residual's weights), and 3D: the y positions.
// Weights are 0 past a wall (the position then is the pair's own); the second
// cell of an odd row's last pair does not exist and has zeros throughout.
// Positions are 16 bits: a block stages at most 3 CC_MAX_PAIRS pairs.
constexpr unsigned CC_NONE = 0xffffu;
__device__ __forceinline__ float cc_pack(unsigned lo, unsigned hi) { return __uint_as_float(lo | (hi << 16)); }
__device__ __forceinline__ unsigned cc_lo(float v) { return __float_as_uint(v) & 0xffffu; }
__device__ __forceinline__ unsigned cc_hi(float v) { return __float_as_uint(v) >> 16; }

// The plan entry of pair t of level l.
__device__ __forceinline__ void cc_plan_pair(const CoarseCycle& cc, int l, int t) {
    const CCLevel& V = cc.lev[l];
    const Lev32& L = V.L;
    const Geo& g = L.g;
    const int nr = V.nr, arith = V.arith, units = g.nz >> V.hz;
    const int hp = V.hp, ny = g.ny, nz = g.nz, P = hp * ny * nz;
    const int row = t / hp, m = t - row * hp, k = row / ny, j = row - k * ny, i = 2 * m;
    const int rank = nr > 1 ? cc_owner(k >> V.hz, units, nr) : 0;
    auto first = [&](int r) { return cc_unit0(r, units, nr) << V.hz; };
    const int k0 = nr > 1 ? first(rank) : 0, k1 = nr > 1 ? first(rank + 1) : nz;
    const int lr = row - ny * k0, p = m + hp * (lr + ny * V.halo);
    const bool two = i + 1 < g.nx;
    const int c0 = (j + k) & 1;                    // colour of cell 2m
    const bool fm = face_minus(i, g.nx, g.bcx), fp = two && face_plus(i + 1, g.nx, g.bcx);
    const bool ym = face_minus(j, ny, g.bcy), yp = face_plus(j, ny, g.bcy);
    const bool zm = face_minus(k, nz, g.bcz), zp = face_plus(k, nz, g.bcz);
    // row steps to the y and z neighbours: in the grid, and among the staged rows
    const int dym = j > 0 ? -1 : ny - 1, dyp = j < ny - 1 ? 1 : 1 - ny;
    const int dzm = k > 0 ? -ny : (nz - 1) * ny, dzp = k < nz - 1 ? ny : (1 - nz) * ny;
    const int szm = nr > 1 ? -ny : dzm, szp = nr > 1 ? ny : dzp;
    float w[6][2], wr[6][2], dv[2], cv[2];         // by cell of the pair; wr: the operator's own weights
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const bool on = b == 0 || two;
        const int e = i + b + g.nx * row;
        const float rc = on ? L.rho[e] : 1.f, ct = on ? L.ct[e] : 1.f;
        const bool has[6] = {on && (b || fm), on && (b ? fp : two), on && ym, on && yp, on && zm, on && zp};
        const int nb[6] = {b || i > 0 ? e - 1 : e + g.nx - 1, i + b + 1 < g.nx ? e + 1 : e + 1 - g.nx,
                           e + g.nx * dym, e + g.nx * dyp, e + g.nx * dzm, e + g.nx * dzp};
        const float c2[3] = {L.c2x, L.c2y, L.c2z};
        float rn[6];
#pragma unroll
        for (int h = 0; h < 6; ++h) {
            rn[h] = has[h] ? L.rho[nb[h]] : Z2_WALL;
            wr[h][b] = has[h] ? face32(rc, rn[h], c2[h >> 1]) : 0.f;
            w[h][b] = wr[h][b];
        }
        float d;
        if (arith == CC_AXIS) {                    // the two faces of an axis from one reciprocal (z2_gs)
            float r[6];
#pragma unroll
            for (int ax = 0; ax < 6; ax += 2) {
                const float am = rc + rn[ax], ap = rc + rn[ax + 1], tr = rcp_hw(am * ap);
                r[ax] = ap * tr;
                r[ax + 1] = am * tr;
            }
            d = fmaf(L.c2z, r[4] + r[5], fmaf(L.c2x, r[0] + r[1], ct));
#pragma unroll
            for (int h = 0; h < 6; ++h) w[h][b] = has[h] ? r[h] : 0.f;
        } else {
            d = ct + ((w[0][b] + w[1][b]) + (w[2][b] + w[3][b])) + (w[4][b] + w[5][b]);
        }
        dv[b] = !on ? 0.f : (arith == CC_INVERSE ? 1.f / d : rcp_hw(d));
        cv[b] = on ? ct : 0.f;
    }
    const int A = c0, B = 1 - c0;                  // the cell of colour 0, of colour 1
    auto pick = [](const float (&v)[2], int b) { return b ? v[1] : v[0]; };
    const unsigned sA = fm ? (m > 0 ? p - 1 : p + hp - 1) : p, sB = fp ? (m + 1 < hp ? p + 1 : p - hp + 1) : p;
    unsigned lo = CC_NONE, hi = CC_NONE;
    if (nr > 1) {
        // rows of the block's first plane are the upper halo of the block
        // before, those of its last plane the lower halo of the block after
        const int before = rank > 0 ? rank - 1 : nr - 1;
        if (k == k0) lo = m + hp * (j + ny * (first(before + 1) - first(before) + 1));
        if (k == k1 - 1) hi = m + hp * j;
    }
    float4* const o = V.plan + t;
    o[0] = make_float4(pick(w[0], A), pick(w[1], A), pick(w[4], A), pick(w[5], A));
    o[P] = make_float4(pick(w[0], B), pick(w[1], B), pick(w[4], B), pick(w[5], B));
    o[2 * P] = make_float4(pick(dv, A), pick(dv, B), c0 ? cc_pack(sB, sA) : cc_pack(sA, sB),
                           cc_pack(zm ? p + hp * szm : p, zp ? p + hp * szp : p));
    o[3 * P] = make_float4(__uint_as_float((unsigned)(i + g.nx * lr) | (two ? 1u << 30 : 0u) | ((unsigned)c0 << 31)),
                           cc_pack(lo, hi), pick(cv, A), pick(cv, B));
    if (cc.lev[0].L.g.ny > 1) {                    // a 3D chain, whatever this level's own ny
        o[4 * P] = make_float4(pick(w[2], A), pick(w[3], A), pick(w[2], B), pick(w[3], B));
        reinterpret_cast<float*>(V.plan + 5 * P)[t] = cc_pack(ym ? p + hp * dym : p, yp ? p + hp * dyp : p);
    } else if (arith == CC_AXIS) {
        o[4 * P] = make_float4(pick(wr[0], A), pick(wr[1], A), pick(wr[4], A), pick(wr[5], A));
        o[5 * P] = make_float4(pick(wr[0], B), pick(wr[1], B), pick(wr[4], B), pick(wr[5], B));
    }
}

// Every pair of the chain: threads t, t + n, ... take the levels' pairs in turn.
__device__ __forceinline__ void cc_plan_range(const CoarseCycle& cc, int t, int n) {
    for (int l = 0; l < cc.nl - (cc.ainv ? 1 : 0); ++l) {
        const int P = cc_pairs(cc.lev[l].L.g);
        for (; t < P; t += n) cc_plan_pair(cc, l, t);
        t -= P;
    }
}

// ---- transfers between levels (threads tid, tid + n, ... of the block) -----------

// The mean over the children of the block's residual of level l, stored as the
// next level's right-hand side in the block that owns it.
template <int NR>
__device__ __forceinline__ void cc_restrict(float* sm, const CoarseCycle& cc, int l, int rank, int tid, int n) {
    const CCLevel &V = cc.lev[l], &W = cc.lev[l + 1];
    const Geo &F = V.L.g, &g = W.L.g;
    const CCLev s = cc_lev(sm, V, rank);
    float* const fc = cc_lev(sm, W, 0).f;
    const int hx = V.hx, hy = V.hy, hz = V.hz, K0 = s.k0 >> hz, cells = g.nx * g.ny * ((s.k1 - s.k0) >> hz);
    for (int e = tid; e < cells; e += n) {
        const int row = cc_div(e, W.ix), I = e - row * g.nx, lk = cc_div(row, W.iy), J = row - lk * g.ny;
        float sum = 0.f;
        for (int c = 0; c <= hz; ++c)
            for (int b = 0; b <= hy; ++b) {
                const float* const r = s.res + (I << hx) + F.nx * (((J << hy) + b) + F.ny * ((lk << hz) + c));
                sum += r[0];
                if (hx) sum += r[1];
            }
        sum *= V.imean;
        if (NR > 1 && V.nr > 1) {
            const int K = K0 + lk, o = cc_block_of(W, K);
            cc_st_remote(cc_remote(fc + I + g.nx * (J + g.ny * (K - cc_first(W, o))), o), sum);
        } else {
            fc[e] = sum;
        }
    }
}

// The block's solution of level l, stored as the correction of level l - 1 in
// the block that owns its children.
template <int NR>
__device__ __forceinline__ void cc_correct(float* sm, const CoarseCycle& cc, int l, int rank, int tid, int n) {
    const CCLevel &V = cc.lev[l], &U = cc.lev[l - 1];
    const Geo& g = V.L.g;
    const CCLev s = cc_lev(sm, V, rank);
    float* const ec = cc_lev(sm, U, 0).res;
    const int cells = g.nx * g.ny * (s.k1 - s.k0);
    for (int e = tid; e < cells; e += n) {
        const int row = cc_div(e, V.ix), i = e - row * g.nx, lk = cc_div(row, V.iy), j = row - lk * g.ny;
        const int k = s.k0 + lk;
        const float v = ((i + j + k) & 1 ? s.x1 : s.x0)[(i >> 1) + V.hp * (row + g.ny * V.halo)];
        if (NR > 1 && U.nr > 1) {
            const int o = cc_block_of(U, k << U.hz);
            cc_st_remote(cc_remote(ec + i + g.nx * (j + g.ny * (k - (cc_first(U, o) >> U.hz))), o), v);
        } else {
            ec[e] = v;
        }
    }
}

// x += P e on the block's cells of level l and their halo copies.
template <bool CL>
__device__ __forceinline__ void cc_prolong(float* sm, const CoarseCycle& cc, int l, int rank, int tid, int n) {
    const CCLevel &V = cc.lev[l], &W = cc.lev[l + 1];
    const Geo &g = V.L.g, &C = W.L.g;
    const CCLev s = cc_lev(sm, V, rank);
    const int hx = V.hx, hy = V.hy, hz = V.hz, ny = g.ny, cells = g.nx * ny * (s.k1 - s.k0);
    const int before = rank > 0 ? rank - 1 : V.nr - 1, after = rank + 1 < V.nr ? rank + 1 : 0;
    const int nbefore = CL ? cc_first(V, before + 1) - cc_first(V, before) : 0;
    for (int e = tid; e < cells; e += n) {
        const int row = cc_div(e, V.ix), i = e - row * g.nx, lk = cc_div(row, V.iy), j = row - lk * ny;
        const int k = s.k0 + lk, m = i >> 1;
        float* const x = ((i + j + k) & 1) ? s.x1 : s.x0;
        float* const p = x + m + V.hp * (row + ny * V.halo);
        const float v = *p + s.res[(i >> hx) + C.nx * ((j >> hy) + C.ny * (lk >> hz))];
        *p = v;
        if (CL && k == s.k0) cc_st_remote(cc_remote(x + m + V.hp * (j + ny * (nbefore + 1)), before), v);
        if (CL && k == s.k1 - 1) cc_st_remote(cc_remote(x + m + V.hp * j, after), v);
    }
}

// ---- smoothing ---------------------------------------------------------------------

// A pair in registers (see the plan).
struct CCPair {
    float wxm[2], wxp[2], wzm[2], wzp[2], wym[2], wyp[2], di[2], f[2];
    float so, z, y;                 // packed positions
    unsigned own;                   // own cell index, bit 30: the second cell exists, bit 31: the first is black
    unsigned lo, hi;                // the neighbouring blocks' halo copies in x0 (0: none)
};

// What a pass over one level does.
enum CCLeg { CC_DOWN, CC_UP, CC_BOTTOM };

// One leg of the cycle on level l, run by every thread that owns pairs (NQ at
// most; CL: by every thread of the cluster, else by `active` threads of one
// block): DOWN, nu1 red-black sweeps from zero, then the residual, restricted;
// UP, the correction added, then nu2 black-red sweeps; BOTTOM, a coarsest
// level without a dense inverse: COARSE_SWEEPS sweep pairs (red-black,
// black-red) from zero.  UP and BOTTOM end with the correction of the finer
// level.  The second of two half-sweeps of one colour in a row changes nothing
// (every value depends on the other colour only) and is left out.
template <int NR, bool CL, bool Y3, int NQ>
__device__ __forceinline__ void cc_leg(float* sm, const CoarseCycle& cc, int l, CCLeg leg, int rank, int tid,
                                       int active) {
    const CCLevel& V = cc.lev[l];
    const Lev32& L = V.L;
    const CCLev s = cc_lev(sm, V, rank);
    const int arith = V.arith, nr = V.nr;
    const int pp = V.hp * L.g.ny, Pt = pp * L.g.nz;      // pairs of a plane, of the level
    const int P = !CL || rank < nr ? pp * (s.k1 - s.k0) : 0;   // pairs of this block
    const int xs = (int)(s.x1 - s.x0);
    const float4* const plan = V.plan + pp * s.k0;
    const int p0 = tid + pp * V.halo;                    // position of the thread's first pair
    CCPair S[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int t = tid + q * CC_THREADS;
        if (t >= P) continue;
        CCPair& T = S[q];
        const float4 a = __ldg(plan + t), b = __ldg(plan + Pt + t), c = __ldg(plan + 2 * Pt + t);
        const float2 d = __ldg(reinterpret_cast<const float2*>(plan + 3 * Pt + t));
        T.wxm[0] = a.x, T.wxp[0] = a.y, T.wzm[0] = a.z, T.wzp[0] = a.w;
        T.wxm[1] = b.x, T.wxp[1] = b.y, T.wzm[1] = b.z, T.wzp[1] = b.w;
        T.di[0] = c.x, T.di[1] = c.y, T.so = c.z, T.z = c.w;
        T.own = __float_as_uint(d.x);
        if (Y3) {
            const float4 y = __ldg(plan + 4 * Pt + t);
            T.wym[0] = y.x, T.wyp[0] = y.y, T.wym[1] = y.z, T.wyp[1] = y.w;
            T.y = __ldg(reinterpret_cast<const float*>(V.plan + 5 * Pt) + pp * s.k0 + t);
        }
        T.lo = T.hi = 0;
        if (CL) {
            const unsigned lo = cc_lo(d.y), hi = cc_hi(d.y);
            if (lo != CC_NONE) T.lo = cc_remote(s.x0 + lo, rank > 0 ? rank - 1 : nr - 1);
            if (hi != CC_NONE) T.hi = cc_remote(s.x0 + hi, rank + 1 < nr ? rank + 1 : 0);
        }
    }
    auto bar = [&]() {
        if (CL) cc_cluster_sync();
        else asm volatile("bar.sync 1, %0;" ::"r"(active) : "memory");
    };
    if (leg == CC_UP) {                            // while the plan's loads are on their way
        if (P) cc_prolong<CL>(sm, cc, l, rank, tid, active);
        bar();
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        if (tid + q * CC_THREADS >= P) continue;
        CCPair& T = S[q];
        const int own = T.own & 0xffffff;
        const float fa = s.f[own], fb = (T.own >> 30) & 1 ? s.f[own + 1] : 0.f;
        const bool black = T.own >> 31;
        T.f[0] = black ? fb : fa;
        T.f[1] = black ? fa : fb;
    }
    auto put = [&](int q, int c, float v) {
        (c ? s.x1 : s.x0)[p0 + q * CC_THREADS] = v;
        if (CL && S[q].lo) cc_st_remote(S[q].lo + 4 * c * xs, v);
        if (CL && S[q].hi) cc_st_remote(S[q].hi + 4 * c * xs, v);
    };
    // the values of the x neighbours of the pair's cell of colour c, minus first
    auto x_nb = [&](int q, int c, const float* o, float& vm, float& vp) {
        const float vi = o[p0 + q * CC_THREADS], vo = o[c ? cc_hi(S[q].so) : cc_lo(S[q].so)];
        const bool second = (c != 0) != (bool)(S[q].own >> 31);
        vm = second ? vi : vo;
        vp = second ? vo : vi;
    };
    // one half-sweep: colour c from the other colour's values
    auto half = [&](auto colour) {
        constexpr int c = decltype(colour)::value;
        const float* const o = c ? s.x0 : s.x1;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            if (tid + q * CC_THREADS >= P) continue;
            const CCPair& T = S[q];
            float xm, xp, num;
            x_nb(q, c, o, xm, xp);
            const float zm = o[cc_lo(T.z)], zp = o[cc_hi(T.z)];
            if (!Y3 && arith == CC_AXIS) {
                num = fmaf(L.c2x, fmaf(T.wxp[c], xp, T.wxm[c] * xm), T.f[c]);
                num = fmaf(L.c2z, fmaf(T.wzp[c], zp, T.wzm[c] * zm), num);
            } else {
                num = fmaf(T.wxm[c], xm, T.f[c]);
                num = fmaf(T.wxp[c], xp, num);
                if (Y3) {
                    num = fmaf(T.wym[c], o[cc_lo(T.y)], num);
                    num = fmaf(T.wyp[c], o[cc_hi(T.y)], num);
                }
                num = fmaf(T.wzm[c], zm, num);
                num = fmaf(T.wzp[c], zp, num);
            }
            put(q, c, num * T.di[c]);
        }
        bar();
    };
    using Redc = std::integral_constant<int, 0>;
    using Black = std::integral_constant<int, 1>;
    if (leg == CC_UP) {
        for (int it = 0; it < cc.nu2; ++it) {
            half(Black{});
            half(Redc{});
        }
        if (P && l > 0) cc_correct<NR>(sm, cc, l, rank, tid, active);
        return;
    }
    // the first half-sweep from x = 0: red cells see zero neighbours
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        if (tid + q * CC_THREADS < P) put(q, 0, S[q].f[0] * S[q].di[0]);
    bar();
    half(Black{});
    const int more = leg == CC_BOTTOM ? COARSE_SWEEPS : cc.nu1;
    for (int it = 1; it < more; ++it) {
        half(Redc{});
        half(Black{});
    }
    if (leg == CC_BOTTOM) {
        half(Redc{});
        if (P && l > 0) cc_correct<NR>(sm, cc, l, rank, tid, active);
        return;
    }
    // residual f - A x of the pair's cells (the operator's own arithmetic)
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int t = tid + q * CC_THREADS;
        if (t >= P) continue;
        CCPair T = S[q];
        const float2 ct = __ldg(reinterpret_cast<const float2*>(plan + 3 * Pt + t) + 1);
        if (!Y3 && arith == CC_AXIS) {             // the sweep's weights lack 2/h^2: take the operator's
            const float4 a = __ldg(plan + 4 * Pt + t), b = __ldg(plan + 5 * Pt + t);
            T.wxm[0] = a.x, T.wxp[0] = a.y, T.wzm[0] = a.z, T.wzp[0] = a.w;
            T.wxm[1] = b.x, T.wxp[1] = b.y, T.wzm[1] = b.z, T.wzp[1] = b.w;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int b = (c != 0) != (bool)(T.own >> 31);
            if (b && !((T.own >> 30) & 1)) continue;
            const float xc = (c ? s.x1 : s.x0)[p0 + q * CC_THREADS];
            const float* const o = c ? s.x0 : s.x1;
            float xm, xp;
            x_nb(q, c, o, xm, xp);
            float y = (c ? ct.y : ct.x) * xc;
            y = fmaf(T.wxm[c], xc - xm, y);
            y = fmaf(T.wxp[c], xc - xp, y);
            if (Y3) {
                y = fmaf(T.wym[c], xc - o[cc_lo(T.y)], y);
                y = fmaf(T.wyp[c], xc - o[cc_hi(T.y)], y);
            }
            y = fmaf(T.wzm[c], xc - o[cc_lo(T.z)], y);
            y = fmaf(T.wzp[c], xc - o[cc_hi(T.z)], y);
            s.res[(T.own & 0xffffff) + b] = T.f[c] - y;
        }
    }
    // the restriction reads the block's own residual only
    if (CL) __syncthreads();
    else bar();
    if (P) cc_restrict<NR>(sm, cc, l, rank, tid, active);
}

// Coarsest level: x = A^-1 f, cc.parts (16, or 1) threads a row of at most 64.
template <int NR>
__device__ __forceinline__ void cc_solve(float* sm, const CoarseCycle& cc, int tid) {
    const int l = cc.nl - 1, parts = cc.parts;
    const CCLevel& V = cc.lev[l];
    const Geo& g = V.L.g;
    const CCLev s = cc_lev(sm, V, 0);
    const int nc = g.N;
    const float* const A = sm + cc.inv;
    for (int r0 = 0; r0 < nc; r0 += CC_THREADS / parts) {
        const int r = r0 + tid / parts, part = tid % parts;
        float v = 0.f;
        if (r < nc)
            for (int c = part; c < nc; c += parts) v = fmaf(A[r * nc + c], s.f[c], v);
        for (int o = parts >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (r < nc && part == 0) {
            const int row = cc_div(r, V.ix), i = r - row * g.nx, k = cc_div(row, V.iy), j = row - k * g.ny;
            ((i + j + k) & 1 ? s.x1 : s.x0)[(i >> 1) + V.hp * row] = v;
        }
    }
    __syncthreads();
    cc_correct<NR>(sm, cc, l, 0, tid, CC_THREADS);
    __syncthreads();
}

// The legs of a cycle in one loop, so that each variant's code exists (and is
// fetched) once: down to the level above a dense inverse, or through the
// unsolved coarsest level, then back up.
template <int NR, bool Y3>
__device__ __forceinline__ void cc_cycle(float* sm, const CoarseCycle& cc, int rank, int tid) {
    const int nl = cc.nl;
    bool alone = false;                            // the step before was the first block's only
    for (int step = 0; step < 2 * nl - 1; ++step) {
        const int l = step < nl ? step : 2 * (nl - 1) - step;
        const CCLeg leg = step >= nl ? CC_UP : (l + 1 < nl ? CC_DOWN : CC_BOTTOM);
        if (NR > 1 && cc.lev[l].nr > 1) {
            if (alone) cc_cluster_sync();
            alone = false;
            cc_leg<NR, true, Y3, CC_PER_SHARED>(sm, cc, l, leg, rank, tid, CC_THREADS);
            cc_cluster_sync();
        } else {
            alone = true;
            if (NR > 1 && rank > 0) continue;
            if (leg == CC_BOTTOM && cc.ainv) {
                cc_solve<NR>(sm, cc, tid);
                continue;
            }
            const int P = cc_pairs(cc.lev[l].L.g), active = min(CC_THREADS, (P + 31) & ~31);
            if (tid < active) {
                if (P <= CC_THREADS) cc_leg<NR, false, Y3, 1>(sm, cc, l, leg, 0, tid, active);
                else cc_leg<NR, false, Y3, CC_PER>(sm, cc, l, leg, 0, tid, active);
            }
            __syncthreads();
        }
    }
}

// The chain's description is copied to shared memory first: read from where
// the launch put it, each level's fields miss the constant cache anew.
template <int NR, bool Y3>
__device__ __forceinline__ void coarse_cycle_block(const CoarseCycle& given) {
    extern __shared__ __align__(16) float cc_sm[];
    __shared__ CoarseCycle cc;
    const int tid = threadIdx.x, rank = NR == 1 ? 0 : cc_rank();
    for (int e = tid; e < (int)(sizeof(CoarseCycle) / sizeof(int)); e += CC_THREADS)
        reinterpret_cast<int*>(&cc)[e] = reinterpret_cast<const int*>(&given)[e];
    __syncthreads();
    const CCLevel& V = cc.lev[0];
    const Geo& g = V.L.g;
    const CCLev s = cc_lev(cc_sm, V, rank);
    const int plane = g.nx * g.ny, own = rank < V.nr ? plane * (s.k1 - s.k0) : 0;
    cc_copy(s.f, cc.f + plane * s.k0, own, tid);
    if (cc.ainv && rank == 0) {
        const int nc = cc.lev[cc.nl - 1].L.g.N;
        cc_copy(cc_sm + cc.inv, cc.ainv, nc * nc, tid);
    }
    // every position a half-sweep reads without a value yet, or never to have
    // one (a missing second cell, a wall's halo), must hold a finite number
    for (int l = 0; l < cc.nl; ++l) {
        const CCLev v = cc_lev(cc_sm, cc.lev[l], rank);
        for (float* x = v.x0 + tid; x < v.f; x += CC_THREADS) *x = 0.f;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (NR > 1) cc_cluster_sync();
    else __syncthreads();
    cc_cycle<NR, Y3>(cc_sm, cc, rank, tid);
    float* const out = cc.x + plane * s.k0;
    for (int e = tid; e < own; e += CC_THREADS) {
        const int row = cc_div(e, V.ix), i = e - row * g.nx, lk = cc_div(row, V.iy), j = row - lk * g.ny;
        out[e] = (((i + j + s.k0 + lk) & 1) ? s.x1 : s.x0)[(i >> 1) + V.hp * (row + g.ny * V.halo)];
    }
}

}  // namespace lm

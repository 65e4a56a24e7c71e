// Float64 kernels: coefficient assembly, the float64 operator, the Jacobi-
// preconditioned conjugate-gradient iteration and the iterative-refinement
// residual/correction.
//
// GB300 executes float64 at 1/64 of the float32 rate, so these kernels are
// bound by float64 issue, not by HBM: they keep the float64 operation count
// per cell minimal (face conductances and the inverse Jacobi diagonal are
// computed once, at assembly; the stencil uses 13 float64 operations per 3D
// cell) and stream each vector once per kernel.
#include <algorithm>

#include "lm_common.cuh"
#include "lm_kernels.h"
#include "lm_tiles.cuh"

namespace lm {

// ---- coefficient assembly (step (v); Eqs. cpoiss, kappapoiss) -------------

// cells i0 .. i1 - 1 (one launch per chunk of planes when the inputs arrive in chunks)
__global__ void __launch_bounds__(NT) k_assemble(AsmArgs a, int i0, int i1) {
    assemble_range(a, i0 + blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, i1);
}

__global__ void __launch_bounds__(NT) k_scale32(int N, float* __restrict__ x, float scale) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) x[i] *= scale;
}

// Inverse Jacobi diagonal 1/(c~ + sum of the cell's face conductances), from
// the assembled faces (the plus face of a cell is its plus-neighbour's minus face).
__global__ void __launch_bounds__(NT) k_jacobi_diag(Geo g, const double* __restrict__ ct,
                                                    const double* __restrict__ gx, const double* __restrict__ gy,
                                                    const double* __restrict__ gz, double* __restrict__ dinv) {
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.N; idx += stride) {
        int i, j, k;
        cell_coords(idx, g, i, j, k);
        const double d = ct[idx] + gx[idx] + gx[nbr_x(idx, i, g).ip] + gy[idx] + gy[nbr_y(idx, j, g).ip] +
                         gz[idx] + gz[nbr_z(idx, k, g).ip];
        dinv[idx] = ircp(d);
    }
}

// ---- the float64 operator --------------------------------------------------

// y = A x; optional partial sums of x^T A x into part slot 0.
__global__ void __launch_bounds__(NT) k_apply64(Geo g, Op64 op, const double* __restrict__ x,
                                                double* __restrict__ y, double* __restrict__ part) {
    __shared__ double sm[32];
    double acc[1] = {0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.N; idx += stride) {
        const double v = apply64_at(idx, g, op, x);
        y[idx] = v;
        acc[0] += x[idx] * v;
    }
    if (part) write_partials<1>(acc, part, sm);
}

// ---- Jacobi-preconditioned CG (float64) ------------------------------------
// Partial-sum slots: 0 p.q, 1 r.r, 2/3 r.z (even/odd iteration), 4 f.f

__global__ void __launch_bounds__(NT) k_pcg_init_res(PcgArgs a, int use_x0) {
    __shared__ double sm[64];
    double acc[2] = {0.0, 0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride) {
        const double fi = a.f[idx];
        const double ri = use_x0 ? fi - apply64_at(idx, a.g, a.op, a.x) : fi;
        a.r[idx] = ri;
        acc[0] += ri * ri;
        acc[1] += fi * fi;
    }
    if (!use_x0) {
        for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride) a.x[idx] = 0.0;
    }
    block_sum<2>(acc, sm);
    if (threadIdx.x == 0) {
        a.part[1 * MAX_PARTIALS + blockIdx.x] = acc[0];
        a.part[4 * MAX_PARTIALS + blockIdx.x] = acc[1];
    }
}

// p = D^-1 r, partial r.z into slot rz_slot.  restart = 0: first call of a
// solve (sets ||f|| and the initial history entry); restart = 1: after a
// failed true-residual check.
__global__ void __launch_bounds__(NT) k_pcg_init_p(PcgArgs a, int rz_slot, int restart) {
    __shared__ double sm[32];
    const double rr = reduce_partials(a.part + 1 * MAX_PARTIALS, gridDim.x, sm);
    double fnorm;
    if (!restart) {
        const double ff = reduce_partials(a.part + 4 * MAX_PARTIALS, gridDim.x, sm);
        fnorm = sqrt(ff);
    } else {
        fnorm = a.st->fnorm;
    }
    const double rel = fnorm > 0.0 ? sqrt(rr) / fnorm : 0.0;
    const bool stop = !(fnorm > 0.0) || rel <= a.st->rtol;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (!restart) {
            a.st->fnorm = fnorm;
            a.hist[0] = rel;
        }
        a.st->rel = rel;
        a.st->converged = stop ? 1 : 0;
        a.st->done = stop ? 1 : 0;
    }
    if (stop) return;
    double acc[1] = {0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride) {
        const double ri = a.r[idx];
        const double zi = a.op.dinv[idx] * ri;
        a.p[idx] = zi;
        acc[0] += ri * zi;
    }
    write_partials<1>(acc, a.part + rz_slot * MAX_PARTIALS, sm);
}

// q = A p, partial p.q (slot 0)
__global__ void __launch_bounds__(NT) k_pcg_apply(PcgArgs a) {
    if (a.st->done) return;
    __shared__ double sm[32];
    double acc[1] = {0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride) {
        const double v = apply64_at(idx, a.g, a.op, a.p);
        a.q[idx] = v;
        acc[0] += a.p[idx] * v;
    }
    write_partials<1>(acc, a.part, sm);
}

// alpha = r.z / p.q; x += alpha p; r -= alpha q; partial r.r and r.z (z = D^-1 r)
__global__ void __launch_bounds__(NT) k_pcg_xr(PcgArgs a, int k) {
    if (a.st->done) return;
    __shared__ double sm[64];
    const double pq = reduce_partials(a.part, gridDim.x, sm);
    const double rz = reduce_partials(a.part + (2 + (k & 1)) * MAX_PARTIALS, gridDim.x, sm);
    if (!(pq > 0.0) || !isfinite(pq) || !isfinite(rz)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.st->status = LM_ERR_BREAKDOWN;
            a.st->done = 1;
        }
        return;
    }
    const double alpha = rz / pq;
    double acc[2] = {0.0, 0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride) {
        const double pi = a.p[idx];
        a.x[idx] += alpha * pi;
        const double ri = a.r[idx] - alpha * a.q[idx];
        a.r[idx] = ri;
        acc[0] += ri * ri;
        acc[1] += ri * (a.op.dinv[idx] * ri);
    }
    block_sum<2>(acc, sm);
    if (threadIdx.x == 0) {
        a.part[1 * MAX_PARTIALS + blockIdx.x] = acc[0];
        a.part[(2 + ((k + 1) & 1)) * MAX_PARTIALS + blockIdx.x] = acc[1];
    }
}

// convergence test; beta = r.z_new / r.z_old; p = D^-1 r + beta p
__global__ void __launch_bounds__(NT) k_pcg_p(PcgArgs a, int k) {
    if (a.st->done) return;
    __shared__ double sm[32];
    const double rr = reduce_partials(a.part + 1 * MAX_PARTIALS, gridDim.x, sm);
    const double rz_new = reduce_partials(a.part + (2 + ((k + 1) & 1)) * MAX_PARTIALS, gridDim.x, sm);
    const double rz_old = reduce_partials(a.part + (2 + (k & 1)) * MAX_PARTIALS, gridDim.x, sm);
    const double rel = sqrt(rr) / a.st->fnorm;
    const bool conv = rel <= a.st->rtol;
    const bool bad = !isfinite(rel) || !isfinite(rz_new) || !(rz_old != 0.0);
    const bool last = k + 1 >= a.max_iter;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.hist[k + 1] = rel;
        a.st->iters = k + 1;
        a.st->rel = rel;
        if (conv) a.st->converged = 1;
        if (bad) a.st->status = LM_ERR_BREAKDOWN;
        if (conv || bad || last) a.st->done = 1;
    }
    if (conv || bad || last) return;
    const double beta = rz_new / rz_old;
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride)
        a.p[idx] = a.op.dinv[idx] * a.r[idx] + beta * a.p[idx];
}

// ---- the same iterations in one cooperative kernel ------------------------------
//
// On a grid of a few hundred thousand cells an iteration's three launches cost
// more than its arithmetic (24 us an iteration on 129 x 97 cells, of which
// 0.5 us float64 work), so k_pcg_run runs iterations k0, k0 + 1, ... until the
// solve is done, or k1, without leaving the GPU.  One block per SM keeps its
// cells' x, r, p, q (and, with at most four cells a thread, the operator's
// coefficients) in registers; only p, which neighbours read, and the block
// sums go through L2.  Three grid barriers an iteration stand where the
// launches ended, one thread a block looking at one counter.  (Sums tagged
// with their iteration and waited for by every thread that adds them, in place
// of two of the barriers, took 34 us an iteration: the looks crowd out the
// stores they wait for.)
//
// Every sum is formed in the order of k_pcg_apply, k_pcg_xr and k_pcg_p
// launched with G blocks (one cell a thread: G = ceil(N / 256)), so the
// iterates are bitwise theirs.  With fewer than one such block per SM its
// warps are dealt out over the SMs (WARPS: sums are kept per warp and added as
// block_sum adds them), because one SM's float64 pipe takes 18 cycles an
// instruction; otherwise block b takes the blocks b, b + gridDim.x, ...
//
// Every wait is bounded: past the limit the waiting block raises the error
// flag, which every block sees at its next look, and all return
// (LM_ERR_TIMEOUT).
//
// 129 x 97 cells: 22.9 -> 11.2 us an iteration, 59 x 17 x 65: 31.1 -> 14.8 us,
// 81 x 49 x 70: 86.4 -> 35.9 us.  What is left on the small grids is latency:
// three round trips to L2, three barriers and a chain of some forty dependent
// float64 steps (operator, sums, quotients).

// bar[0]: arrivals since the launch; bar[1]: a block gave up, after `looks` looks
// of about 1 us.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned& target, unsigned looks) {
    __shared__ int s_ok;
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        int ok = 0;
        for (unsigned n = 0; n < looks; ++n) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (v >= target) {
                ok = 1;
                break;
            }
            if ((n & 255) == 255 && *(volatile unsigned*)(bar + 1)) break;
        }
        if (!ok) atomicExch(bar + 1, 1u);
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// block_sum<Q> of a block of NT threads, the result in thread 0: warps that hold
// only zeros (any = false) and the steps of the last tree that would add zeros
// are left out, which changes no sum.
template <int Q>
__device__ __forceinline__ void pcg_block_sum(double (&v)[Q], bool any, double* smem) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (any)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    if (l == 0)
#pragma unroll
        for (int q = 0; q < Q; ++q) smem[q * 32 + w] = v[q];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = l < NT / 32 ? smem[q * 32 + l] : 0.0;
#pragma unroll
        for (int o = NT / 64; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    }
    __syncthreads();
}

// Sums of the G block partials of the slots (WARPS: of the 8 G warp partials,
// eight a block, added as block_sum's last tree adds them) in the order of
// reduce_partials; the result in thread 0.
template <bool WARPS, int Q>
__device__ __forceinline__ void pcg_totals(const double* part, const int (&slot)[Q], int G, double* smem,
                                           double (&v)[Q]) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const double* const p = part + slot[q] * MAX_PARTIALS;
        v[q] = 0.0;
        for (int t = threadIdx.x; t < G; t += NT) {
            if constexpr (WARPS) {
                double w[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) w[u] = __ldcg(p + 8 * t + u);
                v[q] += ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
            } else {
                v[q] += __ldcg(p + t);
            }
        }
    }
    pcg_block_sum<Q>(v, (int)(threadIdx.x & ~31u) < G, smem);
}
// The thread's values v of unit u (virtual block, or warp) into the slots of part.
template <bool WARPS, int Q>
__device__ __forceinline__ void pcg_partial(double (&v)[Q], int u, double* part, const int (&slot)[Q], double* smem) {
    if constexpr (!WARPS) {
        pcg_block_sum<Q>(v, true, smem);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    }
    if (WARPS ? (threadIdx.x & 31) == 0 : threadIdx.x == 0)
#pragma unroll
        for (int q = 0; q < Q; ++q) part[slot[q] * MAX_PARTIALS + u] = v[q];
}

template <bool WARPS, int K>
__global__ void __launch_bounds__(NT, 1) k_pcg_run(PcgArgs a, int G, int k0, int k1, int from_part,
                                                   unsigned* __restrict__ bar, unsigned looks) {
    constexpr bool KEEP = K <= 4;                   // coefficients in registers
    __shared__ double sm[64];
    // scalars of an iteration: formed by one thread each, since every warp that
    // repeats a division occupies the float64 pipe for it
    __shared__ double s_rr, s_rz, s_alpha, s_beta;
    __shared__ int s_bad, s_stop;
    const Geo& g = a.g;
    const int tid = threadIdx.x, units = WARPS ? 8 * G : G;
    const int u0 = WARPS ? (int)(blockIdx.x + gridDim.x * (tid >> 5)) : (int)blockIdx.x;
    unsigned target = 0;
    // the thread's cells: index (-1: none), neighbours, coefficients, vectors
    int id[K], xm[K], xp[K], ym[K], yp[K], zm[K], zp[K];
    double c[K], wxm[K], wxp[K], wym[K], wyp[K], wzm[K], wzp[K], di[K], x[K], r[K], p[K], q[K];
#pragma unroll
    for (int n = 0; n < K; ++n) {
        const int u = u0 + n * gridDim.x, idx = u < units ? (WARPS ? 32 * u + (tid & 31) : NT * u + tid) : g.N;
        id[n] = idx < g.N ? idx : -1;
        x[n] = r[n] = p[n] = q[n] = 0.0;
        if (id[n] < 0) continue;
        int i, j, k;
        cell_coords(idx, g, i, j, k);
        Nbr nb = nbr_x(idx, i, g);
        xm[n] = nb.im, xp[n] = nb.ip;
        nb = nbr_y(idx, j, g);
        ym[n] = nb.im, yp[n] = nb.ip;
        nb = nbr_z(idx, k, g);
        zm[n] = nb.im, zp[n] = nb.ip;
        if (KEEP) {
            c[n] = a.op.ct[idx], di[n] = a.op.dinv[idx];
            wxm[n] = a.op.gx[idx], wxp[n] = a.op.gx[xp[n]];
            wym[n] = a.op.gy[idx], wyp[n] = a.op.gy[yp[n]];
            wzm[n] = a.op.gz[idx], wzp[n] = a.op.gz[zp[n]];
        }
        x[n] = a.x[idx], r[n] = a.r[idx], p[n] = a.p[idx];
    }
    double rz = from_part ? reduce_partials(a.part + (2 + (k0 & 1)) * MAX_PARTIALS, G, sm) : a.st->scale;
    const double fnorm = a.st->fnorm, rtol = a.st->rtol;
    bool ok = true;
    for (int k = k0; k < k1; ++k) {
        // q = A p, p.q
#pragma unroll
        for (int n = 0; n < K; ++n) {
            const int u = u0 + n * gridDim.x;
            if (u >= units) break;
            double acc[1] = {0.0};
            if (id[n] >= 0) {
                const int idx = id[n];
                const double pc = p[n];
                double y = (KEEP ? c[n] : a.op.ct[idx]) * pc;
                y += (KEEP ? wxm[n] : a.op.gx[idx]) * (pc - __ldcg(a.p + xm[n]));
                y += (KEEP ? wxp[n] : a.op.gx[xp[n]]) * (pc - __ldcg(a.p + xp[n]));
                if (g.ny > 1) {
                    y += (KEEP ? wym[n] : a.op.gy[idx]) * (pc - __ldcg(a.p + ym[n]));
                    y += (KEEP ? wyp[n] : a.op.gy[yp[n]]) * (pc - __ldcg(a.p + yp[n]));
                }
                y += (KEEP ? wzm[n] : a.op.gz[idx]) * (pc - __ldcg(a.p + zm[n]));
                y += (KEEP ? wzp[n] : a.op.gz[zp[n]]) * (pc - __ldcg(a.p + zp[n]));
                q[n] = y;
                acc[0] += pc * y;
            }
            const int sl[1] = {0};
            pcg_partial<WARPS, 1>(acc, u, a.part, sl, sm);
        }
        if (!(ok = grid_barrier(bar, target, looks))) break;
        // alpha, x, r, r.r, r.z
        {
            const int sl[1] = {0};
            double pq[1];
            pcg_totals<WARPS, 1>(a.part, sl, G, sm, pq);
            if (tid == 0) {
                s_bad = !(pq[0] > 0.0) || !isfinite(pq[0]) || !isfinite(rz);
                s_alpha = rz / pq[0];
            }
            __syncthreads();
        }
        if (s_bad) {                                 // the same verdict in every block
            if (blockIdx.x == 0 && tid == 0) {
                a.st->status = LM_ERR_BREAKDOWN;
                a.st->done = 1;
            }
            break;
        }
        const double alpha = s_alpha;
#pragma unroll
        for (int n = 0; n < K; ++n) {
            const int u = u0 + n * gridDim.x;
            if (u >= units) break;
            double acc[2] = {0.0, 0.0};
            if (id[n] >= 0) {
                x[n] += alpha * p[n];
                const double ri = r[n] - alpha * q[n];
                r[n] = ri;
                acc[0] += ri * ri;
                acc[1] += ri * ((KEEP ? di[n] : a.op.dinv[id[n]]) * ri);
            }
            const int sl[2] = {1, 2 + ((k + 1) & 1)};
            pcg_partial<WARPS, 2>(acc, u, a.part, sl, sm);
        }
        if (!(ok = grid_barrier(bar, target, looks))) break;
        // beta, p; the convergence test is formed meanwhile and looked at after
        // the barrier (a p updated past the end is not used)
        {
            const int sl[2] = {1, 2 + ((k + 1) & 1)};
            double t[2];
            pcg_totals<WARPS, 2>(a.part, sl, G, sm, t);
            if (tid == 0) {
                s_rr = t[0];
                s_rz = t[1];
            }
            __syncthreads();
            if (tid == 32) s_beta = s_rz / rz;
            __syncthreads();
        }
        const double rz_new = s_rz, beta = s_beta;
#pragma unroll
        for (int n = 0; n < K; ++n)
            if (id[n] >= 0) {
                p[n] = (KEEP ? di[n] : a.op.dinv[id[n]]) * r[n] + beta * p[n];
                __stcg(a.p + id[n], p[n]);
            }
        if (tid == NT - 1) {
            const double rel = sqrt(s_rr) / fnorm;
            const bool conv = rel <= rtol, bad = !isfinite(rel) || !isfinite(rz_new) || !(rz != 0.0);
            s_stop = conv || bad || k + 1 >= a.max_iter;
            if (blockIdx.x == 0) {
                a.hist[k + 1] = rel;
                a.st->iters = k + 1;
                a.st->rel = rel;
                a.st->scale = rz_new;
                if (conv) a.st->converged = 1;
                if (bad) a.st->status = LM_ERR_BREAKDOWN;
                if (s_stop) a.st->done = 1;
            }
        }
        rz = rz_new;
        if (!(ok = grid_barrier(bar, target, looks)) || s_stop) break;
    }
    if (!ok && tid == 0) {
        a.st->status = LM_ERR_TIMEOUT;
        a.st->done = 1;
    }
#pragma unroll
    for (int n = 0; n < K; ++n)
        if (id[n] >= 0) {
            a.x[id[n]] = x[n];
            a.r[id[n]] = r[n];
            a.q[id[n]] = q[n];
        }
}

// r = f - A x, partial r.r (slot 1): the true residual
__global__ void __launch_bounds__(NT) k_true_residual(PcgArgs a) {
    __shared__ double sm[32];
    double acc[1] = {0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < a.g.N; idx += stride) {
        const double ri = a.f[idx] - apply64_at(idx, a.g, a.op, a.x);
        a.r[idx] = ri;
        acc[0] += ri * ri;
    }
    write_partials<1>(acc, a.part + 1 * MAX_PARTIALS, sm);
}

// Single block: st->rel = sqrt(sum of slot) / st->fnorm (or sets fnorm from slot 4)
__global__ void __launch_bounds__(NT) k_finish_rel(double* part, int G, SolveState* st, int set_fnorm,
                                                   double* hist_entry) {
    __shared__ double sm[32];
    const double rr = reduce_partials(part + 1 * MAX_PARTIALS, G, sm);
    if (set_fnorm) {
        const double ff = reduce_partials(part + 4 * MAX_PARTIALS, G, sm);
        if (threadIdx.x == 0) st->fnorm = sqrt(ff);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double fn = st->fnorm;
        st->rel = fn > 0.0 ? sqrt(rr) / fn : 0.0;
        if (hist_entry) *hist_entry = st->rel;
    }
}

// ---- iterative refinement (float64 residual and correction) ---------------

// r = f - A x in float64, stored as float32 times rscale (a power of two
// that keeps the inner problem's float32 values near unit size, so that the
// products of its dot products neither underflow nor overflow) for the
// inner solve; partial r.r (slot 1) and, with FNORM, f.f (slot 4).
// zero_x: x := 0 first (r = f).
// SC: 0 no scaling; 1 the float32 value scaled (a float multiply by a power
// of two, exact while the unscaled residual is a normal float32 -- the
// launcher asks for it when the residual's expected size is well inside
// float32 range; it saves a float64 multiply a cell on GB300's slow float64
// pipe); 2 scaled in float64 before rounding.
// ZERO: x = 0 (which it sets), so r = f: a kernel of its own, since the stencil's
// registers would leave this one, bound by memory, too few warps (256^3: 130 -> 56 us).
template <bool FNORM, int SC, bool ZERO>
__global__ void __launch_bounds__(NT) k_ir_residual(Geo g, Op64 op, const double* __restrict__ f,
                                                    double* __restrict__ x, float* __restrict__ r32,
                                                    double* __restrict__ part, double rscale) {
    __shared__ double sm[64];
    double acc[2] = {0.0, 0.0};
    const float rs32 = (float)rscale;
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.N; idx += stride) {
        const double fi = f[idx];
        const double ri = ZERO ? fi : fi - apply64_fix(idx, g, op, x);
        if (ZERO) x[idx] = 0.0;
        r32[idx] = SC == 2 ? (float)(ri * rscale) : (SC == 1 ? to_f32(ri) * rs32 : to_f32(ri));
        acc[0] += ri * ri;
        if (FNORM && !ZERO) acc[1] += fi * fi;
    }
    if (ZERO) acc[1] = acc[0];
    block_sum<2>(acc, sm);
    if (threadIdx.x == 0) {
        part[1 * MAX_PARTIALS + blockIdx.x] = acc[0];
        if (FNORM) part[4 * MAX_PARTIALS + blockIdx.x] = acc[1];
    }
}

// Warm-start scaling.  Along a direction x the A-norm error of alpha x is
// least at alpha = f.x / x^T A x (then J(alpha x) = -(f.x)^2 / (2 x^T A x) <= J(0)
// for the energy J(x) = x^T A x / 2 - f.x of the SPD system).  Pass 1: partial
// x^T A x (slot 0) and f.x (slot 1).
__global__ void __launch_bounds__(NT) k_warm_dots(Geo g, Op64 op, const double* __restrict__ f,
                                                  const double* __restrict__ x, double* __restrict__ part) {
    __shared__ double sm[64];
    double acc[2] = {0.0, 0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.N; idx += stride) {
        const double xi = x[idx];
        acc[0] += xi * apply64_at(idx, g, op, x);
        acc[1] += f[idx] * xi;
    }
    write_partials<2>(acc, part, sm);
}

// Pass 2: x *= alpha, with alpha = 0 (drop the warm start) unless f.x > 0
// and x^T A x > 0 are finite.  Every block forms alpha from the partials in
// the same order.
__global__ void __launch_bounds__(NT) k_warm_scale(int N, double* __restrict__ x, const double* part, int G) {
    __shared__ double sm[32];
    const double xax = reduce_partials(part, G, sm);
    const double fx = reduce_partials(part + MAX_PARTIALS, G, sm);
    const double alpha = (fx > 0.0 && xax > 0.0 && isfinite(fx) && isfinite(xax)) ? fx / xax : 0.0;
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride)
        x[idx] = alpha > 0.0 ? alpha * x[idx] : 0.0;
}

// x += e * escale (float32 correction accumulated in float64; escale undoes
// the power-of-two scaling of the inner right-hand side, exactly)
__global__ void __launch_bounds__(NT) k_ir_correct(int N, double* __restrict__ x, const float* __restrict__ e,
                                                   double escale) {
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride)
        x[idx] += to_f64(e[idx]) * escale;
}


// Single block: *out = sum of the G partials of slot `slot`.
__global__ void __launch_bounds__(NT) k_reduce_slot(const double* part, int slot, int G, double* out) {
    __shared__ double sm[32];
    const double v = reduce_partials(part + slot * MAX_PARTIALS, G, sm);
    if (threadIdx.x == 0) *out = v;
}

// ---- float64 flexible CG with the float32 multigrid preconditioner --------
// Slots: 0 p.q, 1 r.r, 5 z.q_old, 6 p.r

// partial z.q_old with z the float32 V-cycle output
__global__ void __launch_bounds__(NT) k_fcg64_zq(int N, const float* __restrict__ z, const double* __restrict__ q,
                                                 double* __restrict__ part, const SolveState* st) {
    if (st->done) return;
    __shared__ double sm[32];
    double acc[1] = {0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride) acc[0] += (double)z[idx] * q[idx];
    write_partials<1>(acc, part + 5 * MAX_PARTIALS, sm);
}

// p = z - (z.q_old / p_old.q_old) p_old
__global__ void __launch_bounds__(NT) k_fcg64_p(int N, const float* __restrict__ z, double* __restrict__ p,
                                                const double* __restrict__ part, int first, const SolveState* st) {
    if (st->done) return;
    __shared__ double sm[32];
    double beta = 0.0;
    if (!first) {
        const double zq = reduce_partials(part + 5 * MAX_PARTIALS, gridDim.x, sm);
        const double pq = reduce_partials(part + 0 * MAX_PARTIALS, gridDim.x, sm);
        beta = -zq / pq;
    }
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride)
        p[idx] = (double)z[idx] + beta * (first ? 0.0 : p[idx]);
}

// q = A p; partials p.q (slot 0), p.r (slot 6)
__global__ void __launch_bounds__(NT) k_fcg64_apply(Geo g, Op64 op, const double* __restrict__ p,
                                                    double* __restrict__ q, const double* __restrict__ r,
                                                    double* __restrict__ part, const SolveState* st) {
    if (st->done) return;
    __shared__ double sm[64];
    double acc[2] = {0.0, 0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.N; idx += stride) {
        const double v = apply64_at(idx, g, op, p);
        q[idx] = v;
        const double pi = p[idx];
        acc[0] += pi * v;
        acc[1] += pi * r[idx];
    }
    block_sum<2>(acc, sm);
    if (threadIdx.x == 0) {
        part[0 * MAX_PARTIALS + blockIdx.x] = acc[0];
        part[6 * MAX_PARTIALS + blockIdx.x] = acc[1];
    }
}

// alpha = p.r / p.q; x += alpha p; r -= alpha q; r32 = r; partial r.r (slot 1)
__global__ void __launch_bounds__(NT) k_fcg64_update(int N, double* __restrict__ x, double* __restrict__ r,
                                                     float* __restrict__ r32, const double* __restrict__ p,
                                                     const double* __restrict__ q, double* __restrict__ part,
                                                     SolveState* st) {
    if (st->done) return;
    __shared__ double sm[32];
    const double pq = reduce_partials(part + 0 * MAX_PARTIALS, gridDim.x, sm);
    const double pr = reduce_partials(part + 6 * MAX_PARTIALS, gridDim.x, sm);
    if (!(pq > 0.0) || !isfinite(pq) || !isfinite(pr)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->status = LM_ERR_BREAKDOWN;
            st->done = 1;
        }
        return;
    }
    const double alpha = pr / pq;
    // the preconditioner's input in float32, scaled by a power of two near
    // 1/rms of the previous residual: flexible CG is invariant under a
    // positive scaling of z, and the scaling keeps the float32 V-cycle's
    // values away from underflow as the residual shrinks
    const double rs = pow2_near_inv(st->rel * st->fnorm * rsqrt((double)N));
    double acc[1] = {0.0};
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride) {
        x[idx] += alpha * p[idx];
        const double ri = r[idx] - alpha * q[idx];
        r[idx] = ri;
        r32[idx] = (float)(ri * rs);
        acc[0] += ri * ri;
    }
    write_partials<1>(acc, part + 1 * MAX_PARTIALS, sm);
}

// r32 = r (float32 copy for the preconditioner)
__global__ void __launch_bounds__(NT) k_to32(int N, const double* __restrict__ r, float* __restrict__ r32) {
    const int stride = gridDim.x * blockDim.x;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += stride) r32[idx] = (float)r[idx];
}

// Single block: st->fnorm = sqrt(sum of slot), st->rel = 1 (start of a solve
// whose reference norm is that of its initial residual).
__global__ void __launch_bounds__(NT) k_set_fnorm(const double* part, int slot, int G, SolveState* st) {
    __shared__ double sm[32];
    const double v = reduce_partials(part + slot * MAX_PARTIALS, G, sm);
    if (threadIdx.x == 0) {
        st->fnorm = sqrt(v);
        st->rel = 1.0;
    }
}

// ---- host launchers ---------------------------------------------------------

void launch_assemble(const Geo& g, int G, cudaStream_t s, const double* a_in, const double* rho_new,
                     const double* cs2, double dt, int raw, const double h[3], const Op64Out& out, AsmFlags* fl,
                     int i0, int i1) {
    count_launches(1);
    k_assemble<<<G, NT, 0, s>>>(asm_args(g, a_in, rho_new, cs2, dt, raw, h, out, fl), i0, i1 < 0 ? g.N : i1);
}
void launch_scale32(int N, int G, cudaStream_t s, float* x, float scale) {
    count_launches(1);
    k_scale32<<<G, NT, 0, s>>>(N, x, scale);
}
void launch_jacobi_diag(const Geo& g, int G, cudaStream_t s, const Op64& op, double* dinv) {
    count_launches(1);
    k_jacobi_diag<<<G, NT, 0, s>>>(g, op.ct, op.gx, op.gy, op.gz, dinv);
}
void launch_apply64(const Geo& g, int G, cudaStream_t s, const Op64& op, const double* x, double* y,
                    double* part) {
    count_launches(1);
    k_apply64<<<G, NT, 0, s>>>(g, op, x, y, part);
}
void launch_pcg_init(const PcgArgs& a, int G, cudaStream_t s, int use_x0) {
    count_launches(1);
    k_pcg_init_res<<<G, NT, 0, s>>>(a, use_x0);
    count_launches(1);
    k_pcg_init_p<<<G, NT, 0, s>>>(a, 2, 0);
}
void launch_pcg_init_p(const PcgArgs& a, int G, cudaStream_t s, int rz_slot, int restart) {
    count_launches(1);
    k_pcg_init_p<<<G, NT, 0, s>>>(a, rz_slot, restart);
}
void launch_pcg_xr(const PcgArgs& a, int G, cudaStream_t s, int k) {
    count_launches(1);
    k_pcg_xr<<<G, NT, 0, s>>>(a, k);
}
void launch_pcg_p(const PcgArgs& a, int G, cudaStream_t s, int k) {
    count_launches(1);
    k_pcg_p<<<G, NT, 0, s>>>(a, k);
}
void launch_pcg_restart(const PcgArgs& a, int G, cudaStream_t s, int k) {
    count_launches(1);
    k_pcg_init_p<<<G, NT, 0, s>>>(a, 2 + (k & 1), 1);
}
void launch_pcg_iter(const PcgArgs& a, int G, cudaStream_t s, int k) {
    count_launches(1);
    k_pcg_apply<<<G, NT, 0, s>>>(a);
    count_launches(1);
    k_pcg_xr<<<G, NT, 0, s>>>(a, k);
    count_launches(1);
    k_pcg_p<<<G, NT, 0, s>>>(a, k);
}
// The line lies where the kernel's registers end: eight cells a thread of one
// block per SM (311,296 cells on 152 SMs), which is also where a launch's
// blocks stop having one cell a thread.  Larger grids are bound by the float64
// pipe, not by the launches.
bool pcg_run_fits(int N, int G, int nsm) { return (long long)G * NT >= N && G <= 8 * nsm; }
int launch_pcg_run(const PcgArgs& a, int G, int nsm, cudaStream_t s, int k0, int k1, int from_part, unsigned* bar,
                   unsigned looks) {
    if (cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), s) != cudaSuccess) return LM_ERR_CUDA;
    const void* f;
    int blocks = nsm;
    if (G < nsm) {
        f = (const void*)k_pcg_run<true, 1>;
        blocks = std::min(nsm, 2 * G);               // four warps with cells a block: 11.2 us, one or two: 12.3
    } else if (G <= 2 * nsm) f = (const void*)k_pcg_run<false, 2>;
    else if (G <= 4 * nsm) f = (const void*)k_pcg_run<false, 4>;
    else f = (const void*)k_pcg_run<false, 8>;
    PcgArgs args = a;
    void* av[] = {&args, &G, &k0, &k1, &from_part, &bar, &looks};
    if (cudaLaunchCooperativeKernel(f, dim3(blocks), dim3(NT), av, 0, s) != cudaSuccess) {
        cudaGetLastError();
        return LM_ERR_CUDA;
    }
    count_launches(1);
    return LM_OK;
}
void launch_true_residual(const PcgArgs& a, int G, cudaStream_t s) {
    count_launches(1);
    k_true_residual<<<G, NT, 0, s>>>(a);
    count_launches(1);
    k_finish_rel<<<1, NT, 0, s>>>(a.part, G, a.st, 0, nullptr);
}
void launch_ir_residual(const Geo& g, int G, cudaStream_t s, const Op64& op, const double* f, double* x,
                        float* r32, double* part, int zero_x, SolveState* st, int set_fnorm, double* hist_entry,
                        double rscale) {
    count_launches(1);
    // rscale near 1/rms(r): the residual's size is about 1/rscale, a normal
    // float32 (with room for small entries) when rscale is within 2^+-90
    const int sc = rscale == 1.0 ? 0 : (rscale >= 0x1p-90 && rscale <= 0x1p90 ? 1 : 2);
#define LM_IRR(F, SC, Z) k_ir_residual<F, SC, Z><<<G, NT, 0, s>>>(g, op, f, x, r32, part, rscale)
#define LM_IRR_SC(F, Z) \
    do {                \
        if (sc == 0) LM_IRR(F, 0, Z); else if (sc == 1) LM_IRR(F, 1, Z); else LM_IRR(F, 2, Z); \
    } while (0)
    if (zero_x) {
        if (set_fnorm) LM_IRR_SC(true, true); else LM_IRR_SC(false, true);
    } else {
        if (set_fnorm) LM_IRR_SC(true, false); else LM_IRR_SC(false, false);
    }
#undef LM_IRR_SC
#undef LM_IRR
    count_launches(1);
    k_finish_rel<<<1, NT, 0, s>>>(part, G, st, set_fnorm, hist_entry);
}
void launch_warm_scale(const Geo& g, int G, cudaStream_t s, const Op64& op, const double* f, double* x,
                       double* part) {
    count_launches(2);
    k_warm_dots<<<G, NT, 0, s>>>(g, op, f, x, part);
    k_warm_scale<<<G, NT, 0, s>>>(g.N, x, part, G);
}
void launch_ir_correct(int N, int G, cudaStream_t s, double* x, const float* e, double escale) {
    count_launches(1);
    k_ir_correct<<<G, NT, 0, s>>>(N, x, e, escale);
}
void launch_reduce_rel(double* part, int G, cudaStream_t s, SolveState* st, double* hist_entry) {
    count_launches(1);
    k_finish_rel<<<1, NT, 0, s>>>(part, G, st, 0, hist_entry);
}

void launch_reduce_slot(const double* part, int slot, int G, cudaStream_t s, double* out) {
    count_launches(1);
    k_reduce_slot<<<1, NT, 0, s>>>(part, slot, G, out);
}
void launch_fcg64_iter_a(int N, int G, cudaStream_t s, const float* z, const double* q, double* part, int first,
                         double* p, const SolveState* st) {
    if (!first) {
        count_launches(1);
        k_fcg64_zq<<<G, NT, 0, s>>>(N, z, q, part, st);
    }
    count_launches(1);
    k_fcg64_p<<<G, NT, 0, s>>>(N, z, p, part, first, st);
}
void launch_fcg64_iter_b(const Geo& g, int G, cudaStream_t s, const Op64& op, double* x, double* r, float* r32,
                         const double* p, double* q, double* part, SolveState* st) {
    count_launches(1);
    k_fcg64_apply<<<G, NT, 0, s>>>(g, op, p, q, r, part, st);
    count_launches(1);
    k_fcg64_update<<<G, NT, 0, s>>>(g.N, x, r, r32, p, q, part, st);
    count_launches(1);
    k_finish_rel<<<1, NT, 0, s>>>(part, G, st, 0, nullptr);
}
void launch_set_fnorm(const double* part, int slot, int G, cudaStream_t s, SolveState* st) {
    count_launches(1);
    k_set_fnorm<<<1, NT, 0, s>>>(part, slot, G, st);
}
void launch_to32(int N, int G, cudaStream_t s, const double* r, float* r32) {
    count_launches(1);
    k_to32<<<G, NT, 0, s>>>(N, r, r32);
}

}  // namespace lm

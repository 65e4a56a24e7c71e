// The explicit parts of one fractional step around the pressure solve
// (Sec. 2.4), in float64:
//
//   lm_advect      steps (i)-(iii): face velocities of Eq. step1 from the
//                  cell momenta, the modified flux F~ = (rho, rho c, rho u,
//                  e) u_{i+1/2} evaluated with the upwind side's MUSCL state
//                  (minmod-limited slope; the paper's CPM/MENO reconstruction
//                  is not reproduced in its text), and the explicit update
//                  q^{new} = q^n - dt d(F~)/dx summed over the axes;
//   lm_eos_ideal   step (ix): P = (gamma - 1)(e - |rho u|^2 / (2 rho)) and
//                  c_s^2 = gamma P / rho for the next step's c~.
//
// A wall face carries no flux and a cell next to a wall has zero slope (its
// outer neighbour does not exist); periodic axes wrap.
//
// The float64 pipe bounds it on GB300 (one warp instruction per 18.5 cycles an
// SM), so every difference, slope and face flux is formed once, in one pass an
// axis, and every comparison and quotient runs on the integer pipe
// (lm_intfp.cuh): five float64 instructions a quantity, cell and axis where one
// thread a cell, forming both faces of every axis, took 22.  Along y and z a
// thread marches up a chunk of a column and keeps the last face in registers;
// along x the lanes of a warp hold successive cells and pass differences, slopes
// and fluxes by shuffles.  The passes after the first add to the outputs.
// Five quantities on 96^3 791 -> 175 us, on 256^2 52 -> 21 us.
#include <cuda_runtime.h>

#include <cstdio>

#include "../../include/lowmach.h"
#include "lm_common.cuh"
#include "lm_kernels.h"

namespace {

constexpr int MAXQ = 6;       // rho, rho u (3), e, rho c

struct AdvGeo {
    int n;                    // cells along the pass's axis
    int stride;               // between them
    int wall;
    int rows;                 // columns of the axis: N / n
    int inner, outer;         // column q starts at (q / inner) outer + q % inner
    int L;                    // cells a thread (y and z)
    double dt, rh;            // rh = 1 / h
};

struct AdvIO {
    const double* q[MAXQ];    // rho, m_x, m_y, m_z, e, rho c
    double* out[MAXQ];
};

__device__ __forceinline__ double minmod(double a, double b) {
    return __longlong_as_double((long long)lm::minmod_bits(lm::dbits(a), lm::dbits(b)));
}

// offset along an axis of the cell at position d in [-2, n + 1]: wrapped on a
// periodic axis, clamped on a wall axis (clamped values are never used: wall
// cells have zero slope and the wall face no flux)
__device__ __forceinline__ int along(int d, int n, int wall) {
    if (d < 0) return wall ? 0 : d + n;
    if (d >= n) return wall ? n - 1 : d - n;
    return d;
}

// dt u of the minus face of the cell at position c (Eq. step1), cells m and c
__device__ __forceinline__ double face_w(const AdvGeo& G, int c, double rm, double rc, double mm, double mc) {
    return G.wall && (c == 0 || c == G.n) ? 0.0 : G.dt * lm::idiv(mm + mc, rm + rc);
}
// dt times a quantity's flux through it: the upwind side's value at the face
__device__ __forceinline__ double face_flux(double w, double xm, double sm, double xc, double sc) {
    const bool up = (int64_t)lm::dbits(w) > 0;
    return fma(up ? 0.5 : -0.5, up ? sm : sc, up ? xm : xc) * w;
}
__device__ __forceinline__ bool flat_at(const AdvGeo& G, int c) { return G.wall && (c <= 0 || c >= G.n - 1); }

// The pass along x, the first where nx > 1.  A row's items are its positions -1 ..
// n + 1; a warp takes 32 successive items of all rows and writes the 29 whose
// difference, slopes and fluxes its lanes hold.
template <int NQ>
__global__ void __launch_bounds__(lm::NT) k_advect_x(AdvGeo G, AdvIO io) {
    constexpr int OUT = 29;
    const int lane = threadIdx.x & 31;
    const uint64_t m = (uint64_t)G.n + 3, items = (uint64_t)G.rows * m;
    const uint64_t warps = (items + OUT - 1) / OUT, step = (uint64_t)gridDim.x * (lm::NT / 32);
    const bool small = items + 64 < (1ull << 32);
    for (uint64_t w0 = (uint64_t)blockIdx.x * (lm::NT / 32) + threadIdx.x / 32; w0 < warps; w0 += step) {
        uint64_t it = w0 * OUT + lane;
        const bool in = it < items;
        if (!in) it = items - 1;
        const int row = small ? (int)((uint32_t)it / (uint32_t)m) : (int)(it / m);
        const int c = (int)(it - (uint64_t)row * m) - 1;
        const int base = row * G.n, ic = base + along(c, G.n, G.wall), im = base + along(c - 1, G.n, G.wall);
        double xc[NQ], xm[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) xc[q] = io.q[q][ic], xm[q] = io.q[q][im];
        const double w = face_w(G, c, xm[0], xc[0], xm[1], xc[1]);
        const bool flat = flat_at(G, c), put = in && lane >= 1 && lane <= OUT && c >= 0 && c < G.n;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const double d = xc[q] - xm[q], dn = __shfl_down_sync(~0u, d, 1);
            const double s = flat ? 0.0 : minmod(d, dn), sm = __shfl_up_sync(~0u, s, 1);
            const double f = face_flux(w, xm[q], sm, xc[q], s), fn = __shfl_down_sync(~0u, f, 1);
            if (put) io.out[q][ic] = fma(G.rh, f - fn, xc[q]);
        }
    }
}

// The pass along y (A = 1) or z (A = 2): a thread takes L cells of a column.
template <int A, int NQ, bool FIRST>
__global__ void __launch_bounds__(128) k_advect_col(AdvGeo G, AdvIO io) {
    const int q0 = blockIdx.x * blockDim.x + threadIdx.x;
    if (q0 >= G.rows) return;
    const int col = q0 / G.inner * G.outer + q0 % G.inner;
    const int c0 = blockIdx.y * G.L, c1 = min(c0 + G.L, G.n);
    double xm[NQ], xc[NQ], d[NQ], s[NQ], f[NQ];
    {
        const int i0 = col + along(c0 - 2, G.n, G.wall) * G.stride, i1 = col + along(c0 - 1, G.n, G.wall) * G.stride,
                  i2 = col + c0 * G.stride;
        const bool flat = flat_at(G, c0 - 1);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            xm[q] = io.q[q][i1];
            xc[q] = io.q[q][i2];
            d[q] = xc[q] - xm[q];
            s[q] = flat ? 0.0 : minmod(xm[q] - io.q[q][i0], d[q]);
        }
    }
    double xn[NQ], o[NQ];                                  // the next face's loads, a face ahead
    auto fetch = [&](int c) {
        const int in = col + along(c + 1, G.n, G.wall) * G.stride, im = col + (c - 1) * G.stride;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            xn[q] = io.q[q][in];
            if (!FIRST && c > c0) o[q] = io.out[q][im];
        }
    };
    fetch(c0);
    for (int c = c0; c <= c1; ++c) {                       // the minus face of cell c, the update of cell c - 1
        const int im = col + (c - 1) * G.stride;
        const double w = face_w(G, c, xm[0], xc[0], xm[1 + A], xc[1 + A]);
        const bool flat = flat_at(G, c);
        double y[NQ];
#pragma unroll
        for (int q = 0; q < NQ; ++q) y[q] = FIRST ? xm[q] : o[q];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const double dn = xn[q] - xc[q];
            const double sc = flat ? 0.0 : minmod(d[q], dn);
            const double fc = face_flux(w, xm[q], s[q], xc[q], sc);
            if (c > c0) y[q] = fma(G.rh, f[q] - fc, y[q]);
            xm[q] = xc[q];
            xc[q] = xn[q];
            d[q] = dn;
            s[q] = sc;
            f[q] = fc;
        }
        if (c < c1) fetch(c + 1);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (c > c0) io.out[q][im] = y[q];
    }
}

// Cells a thread of a column pass: the first face and slopes cost about one more
// cell, so long chunks, but no longer than leaves every SM six warps (one against
// two and four cells: 96 x 56 17, 19 and 23 us; two against four: 256^2 25 and 27;
// nine against four: 32 x 96 x 120 132 and 150).
int column_cells(long long N, int n) {
    const long long l = N / (152 * 170);
    int L = (int)(l < 1 ? 1 : (l > 16 ? 16 : l));
    L = L < n / 65535 + 1 ? n / 65535 + 1 : L;            // (a grid holds 65535 of them)
    const int chunks = (n + L - 1) / L;
    return (n + chunks - 1) / chunks;
}

template <int NQ>
void launch_advect(const int n[3], const double rh[3], const int wall[3], double dt, const AdvIO& io, cudaStream_t s) {
    const long long N = (long long)n[0] * n[1] * n[2];
    bool first = true;
    for (int a = 0; a < 3; ++a) {
        if (n[a] == 1) continue;
        AdvGeo G{};
        G.n = n[a];
        G.wall = wall[a];
        G.rows = (int)(N / n[a]);
        G.stride = a == 0 ? 1 : (a == 1 ? n[0] : n[0] * n[1]);
        G.inner = G.stride;
        G.outer = a == 1 ? n[0] * n[1] : 0;
        G.dt = dt;
        G.rh = rh[a];
        lm::count_launches(1);
        if (a == 0) {
            const unsigned long long warps = ((unsigned long long)G.rows * (G.n + 3) + 28) / 29, b = (warps + 7) / 8;
            k_advect_x<NQ><<<(unsigned)(b > 152 * 64 ? 152 * 64 : b), lm::NT, 0, s>>>(G, io);
        } else {
            G.L = column_cells(N, G.n);
            const dim3 grid((unsigned)((G.rows + 127) / 128), (unsigned)((G.n + G.L - 1) / G.L));
            if (a == 1 && first) k_advect_col<1, NQ, true><<<grid, 128, 0, s>>>(G, io);
            else if (a == 1) k_advect_col<1, NQ, false><<<grid, 128, 0, s>>>(G, io);
            else if (first) k_advect_col<2, NQ, true><<<grid, 128, 0, s>>>(G, io);
            else k_advect_col<2, NQ, false><<<grid, 128, 0, s>>>(G, io);
        }
        first = false;
    }
    if (first)                                             // one cell: nothing flows
        for (int q = 0; q < NQ; ++q) cudaMemcpyAsync(io.out[q], io.q[q], sizeof(double) * N, cudaMemcpyDeviceToDevice, s);
}

__global__ void __launch_bounds__(lm::NT) k_eos_ideal(int N, double gamma, const double* __restrict__ rho,
                                                      const double* __restrict__ mom,
                                                      const double* __restrict__ e, double* __restrict__ p,
                                                      double* __restrict__ cs2) {
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += gridDim.x * blockDim.x) {
        const double r = rho[idx];
        const double mx = mom[idx], my = mom[(size_t)N + idx], mz = mom[2 * (size_t)N + idx];
        const double kin = lm::idiv(0.5 * (mx * mx + my * my + mz * mz), r);
        const double pi = (gamma - 1.0) * (e[idx] - kin);
        p[idx] = pi;
        if (cs2) cs2[idx] = lm::idiv(gamma * pi, r);
    }
}

int blocks_for(long long N) {
    long long b = (N + lm::NT - 1) / lm::NT;
    return (int)(b < 1 ? 1 : (b > 8 * 152 ? 8 * 152 : b));
}

int finish(const char* what) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        fprintf(stderr, "lowmach: %s: %s\n", what, cudaGetErrorString(e));
        return LM_ERR_CUDA;
    }
    return LM_OK;
}

}  // namespace

extern "C" {

int lm_advect(int ndim, const int64_t n[3], const double h[3], const int bc[3], double dt, const double* rho,
              const double* mom, const double* e, const double* rho_c, double* rho_new, double* mom_star,
              double* e_star, double* rho_c_new, void* stream) {
    if (!n || !h || !bc || (ndim != 2 && ndim != 3) || !rho || !mom || !e || !rho_new || !mom_star || !e_star ||
        (!rho_c) != (!rho_c_new) || !(dt >= 0.0 && dt < 1e300))
        return LM_ERR_INVALID_ARG;
    for (int a = 0; a < 3; ++a)
        if (n[a] < 1 || !(h[a] > 0.0) || (bc[a] != LM_BC_PERIODIC && bc[a] != LM_BC_NEUMANN)) return LM_ERR_INVALID_ARG;
    if ((ndim == 2 && n[1] != 1) || (long long)n[0] * n[1] * n[2] >= (1LL << 31)) return LM_ERR_INVALID_ARG;
    const int nn[3] = {(int)n[0], (int)n[1], (int)n[2]};
    double rh[3];
    int wall[3];
    for (int a = 0; a < 3; ++a) {
        wall[a] = bc[a] == LM_BC_NEUMANN;
        rh[a] = 1.0 / h[a];
    }
    const int nq = rho_c ? 6 : 5;
    const size_t N = (size_t)nn[0] * nn[1] * nn[2];
    // the outputs must not overlap the inputs (every thread reads neighbours)
    const double* ins[MAXQ] = {rho, mom, mom + N, mom + 2 * N, e, rho_c};
    double* outs[MAXQ] = {rho_new, mom_star, mom_star + N, mom_star + 2 * N, e_star, rho_c_new};
    for (int q = 0; q < nq; ++q)
        for (int r = 0; r < nq; ++r)
            if (outs[q] < ins[r] + N && ins[r] < outs[q] + N) return LM_ERR_INVALID_ARG;
    AdvIO io{};
    for (int q = 0; q < nq; ++q) {
        io.q[q] = ins[q];
        io.out[q] = outs[q];
    }
    if (nq == 6)
        launch_advect<6>(nn, rh, wall, dt, io, (cudaStream_t)stream);
    else
        launch_advect<5>(nn, rh, wall, dt, io, (cudaStream_t)stream);
    return finish("lm_advect");
}

int lm_eos_ideal(int64_t n_cells, double gamma, const double* rho, const double* mom, const double* e, double* p,
                 double* cs2, void* stream) {
    if (n_cells < 1 || n_cells >= (1LL << 31) || !(gamma > 1.0) || !rho || !mom || !e || !p) return LM_ERR_INVALID_ARG;
    lm::count_launches(1);
    k_eos_ideal<<<blocks_for(n_cells), lm::NT, 0, (cudaStream_t)stream>>>((int)n_cells, gamma, rho, mom, e, p, cs2);
    return finish("lm_eos_ideal");
}

}  // extern "C"

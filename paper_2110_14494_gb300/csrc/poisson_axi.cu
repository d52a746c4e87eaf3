// Axisymmetric Poisson solve (Sec. 2.5 in the paper's axisymmetric geometry,
// Sec. 2.1.2 for the ring cells): -(1/r) d/dr (r dphi/dr) - d2phi/dz2 = rho /
// eps0 on a cell-centred (r, z) mesh, cells i = 0..nr-1 at r_i = (i + 1/2) h
// from the axis, k = 0..nz-1 along z, square cells of side h.
//
// Each row is the flux balance of a ring cell divided by 2 pi h (symmetric,
// positive definite): with r in units of h the face coefficients are i
// (inner radial face, 0 on the axis), i + 1 (outer radial face) and i + 1/2
// (the two axial faces), and the right-hand side is (i + 1/2) h^2 rho / eps0.
// Boundaries: the outer cylinder homogeneous Neumann (no flux), the z faces
// Dirichlet plates v_lo, v_hi (ghost 2 v - phi), cells of the electrode mask
// held at v_mask.  E = -grad(phi) by central differences at cell centres
// (mirror at the axis and the outer cylinder).
//
// Solver: flexible CG in float64 preconditioned by one float64 V(2,2)-cycle
// of red-black Gauss-Seidel on the same operator re-discretised on every
// level (coarse cells twice as wide; a coarse cell is held at zero if any
// child is masked).  The coarse right-hand side is half the sum of the four
// children's residuals: residuals are fluxes divided by 2 pi h, and the
// coarse cell's fluxes are the sums of its children's, divided by 2 pi (2h).
//
// What bounds it: the double pipe (a warp's operation takes 18 clocks of its
// multiprocessor) on the fine level, the chain of kernels below it.  So every
// lane of a half-sweep updates a cell, a cell costs six double operations
// (reciprocal diagonals by column instead of a division, face coefficients
// formed once a thread), the first sweep from zero is one kernel, red cells
// alone are interpolated and restricted, levels of 1024 cells and fewer are
// one block, and a CG iteration adds two kernels.
#include <math.h>

#include "common.cuh"
#include "graph_util.cuh"
#include "poisson_axi.cuh"
#include "../../include/picmcc.h"

namespace pic {

namespace {

constexpr int AX = 32, AZ = 8;
const dim3 kABlk(AX, AZ, 1);
enum { A_B2 = 0, A_R2, A_RHO, A_GAM, A_T1, A_T2, A_ALPHA, A_BETA, A_N };

dim3 agrid(int nr, int nz) { return dim3((nr + AX - 1) / AX, (nz + AZ - 1) / AZ); }
// Kernels whose threads walk kRows planes; in the red-black ones a thread takes one cell of each pair in r.
constexpr int kRows = 4;
dim3 agrid_rows(int nr, int nz) { return dim3((nr + AX - 1) / AX, (nz + AZ * kRows - 1) / (AZ * kRows)); }
// Red-black kernels: kRows planes a thread on levels of 2^17 cells and more (the loads of four cells in flight),
// one below (more blocks: 64 x 64 cells would occupy two multiprocessors).
bool deep(int nr, int nz) { return (long long)nr * nz >= 1 << 17; }
dim3 agrid_half(int nr, int nz) {
    return deep(nr, nz) ? agrid_rows((nr + 1) / 2, nz) : agrid((nr + 1) / 2, nz);
}

// Sums NV per-thread values over the grid: each block stores its sums, the
// last one to arrive adds them in a fixed order, leaves the totals in tot[]
// of its thread 0 and returns true there; the counter is reset.
template <int NV>
__device__ bool axi_sums(const double (&v)[NV], double* part, unsigned* ctr, double (&tot)[NV]) {
    __shared__ double red[NV][32];
    __shared__ int last;
    const int t = threadIdx.x + threadIdx.y * blockDim.x, lane = t & 31, w = t >> 5;
    const int nthr = blockDim.x * blockDim.y, nw = nthr >> 5;
    const unsigned b = blockIdx.x + gridDim.x * blockIdx.y, nb = gridDim.x * gridDim.y;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double x = v[q];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
        if (lane == 0) red[q][w] = x;
    }
    __syncthreads();
    if (t == 0) {
        for (int q = 0; q < NV; ++q) {
            double s = 0.0;
            for (int x = 0; x < nw; ++x) s += red[q][x];
            part[(size_t)b * NV + q] = s;
        }
        __threadfence();
        last = atomicAdd(ctr, 1u) == nb - 1 ? 1 : 0;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double s = 0.0;
        for (unsigned x = t; x < nb; x += nthr) s += __ldcg(part + (size_t)x * NV + q);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        __syncthreads();
        if (lane == 0) red[q][w] = s;
        __syncthreads();
        if (t == 0) {
            double a = 0.0;
            for (int x = 0; x < nw; ++x) a += red[q][x];
            tot[q] = a;
        }
    }
    if (t == 0) *ctr = 0u;
    return t == 0;
}

// Face coefficients of cell (i, k): inner, outer radial and axial.
struct Coef {
    double ci, co, cz;
};
__device__ __forceinline__ Coef coef(int i, int nr) {
    return Coef{(double)i, i + 1 < nr ? (double)(i + 1) : 0.0, (double)i + 0.5};
}
__device__ __forceinline__ double diag_of(const Coef& c, int k, int nz) {
    return c.ci + c.co + 2.0 * c.cz + (k == 0 ? c.cz : 0.0) + (k == nz - 1 ? c.cz : 0.0);
}
// Weighted neighbour sum of the correction e (zero on masked cells and in
// the homogeneous ghosts: Dirichlet ghost -e is in the diagonal).
__device__ __forceinline__ double nb_e(const double* e, int i, int k, int nr, int nz, const Coef& c) {
    const int q = k * nr + i;
    double s = 0.0;
    if (i > 0) s += c.ci * e[q - 1];
    if (i + 1 < nr) s += c.co * e[q + 1];
    if (k > 0) s += c.cz * e[q - nr];
    if (k + 1 < nz) s += c.cz * e[q + nr];
    return s;
}

#define ACELL                                          \
    const int i = blockIdx.x * AX + threadIdx.x;      \
    const int k = blockIdx.y * AZ + threadIdx.y;      \
    const bool in = i < nr && k < nz;                 \
    const int c = in ? k * nr + i : 0;

__global__ void k_axi_copy_mask(const uint8_t* m, uint8_t* out, int n) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) out[c] = m ? (m[c] ? 1 : 0) : 0;
}

__global__ void k_axi_restrict_mask(const uint8_t* __restrict__ m, int nr, int nz, uint8_t* __restrict__ mc) {
    const int cr = nr / 2, cz = nz / 2;
    const int I = blockIdx.x * AX + threadIdx.x, K = blockIdx.y * AZ + threadIdx.y;
    if (I >= cr || K >= cz) return;
    uint8_t v = 0;
    for (int d = 0; d < 4; ++d) v |= m[(2 * K + (d >> 1)) * nr + 2 * I + (d & 1)];
    mc[K * cr + I] = v ? 1 : 0;
}

__global__ void k_axi_rdiag(int nr, int nz, double* __restrict__ rd) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nr) return;
    const Coef c = coef(i, nr);
    rd[i] = 1.0 / diag_of(c, 1, 3);
    rd[nr + i] = 1.0 / diag_of(c, 0, nz);
}

// b and r = b - A phi with the boundary values; ||b||^2, ||r||^2; electrode
// cells get phi = v_mask, r = 0.  b from the charge density, or from the
// fixed-point charges combined as integers (exact) and converted once: the
// ring volume pi (2 i + 1) h^3 cancels against the factor i + 1/2.
template <bool FIXED>
__global__ void __launch_bounds__(AX * AZ) k_axi_resid(double* __restrict__ phi, const AxiCharge rho,
                                                       const uint8_t* __restrict__ m, int nr, int nz, double h2e,
                                                       double v_lo, double v_hi, double v_mask, double* __restrict__ r,
                                                       double* __restrict__ g0, double* part, unsigned* ctr, double* sc) {
    const int i = blockIdx.x * AX + threadIdx.x, k0 = (blockIdx.y * AZ + threadIdx.y) * kRows;
    double acc[2] = {0.0, 0.0};
    if (i < nr) {
        const Coef cf = coef(i, nr);
        const double wr = cf.cz * h2e;
#pragma unroll
        for (int d = 0; d < kRows; ++d) {
            const int k = k0 + d, c = k * nr + i;
            if (k >= nz) break;
            if (m[c]) {
                phi[c] = v_mask;
                r[c] = 0.0;
                g0[c] = 0.0;
                continue;
            }
            const double pc = phi[c];
            double b = FIXED ? rho.scale * (double)(rho.qp[c] - rho.qn[c] - rho.qe[c]) : wr * rho.rho[c];
            double s = b;
            auto face = [&](int q, double w) {
                if (m[q]) { b += w * v_mask; s += w * (v_mask - pc); }
                else s += w * (phi[q] - pc);
            };
            if (i > 0) face(c - 1, cf.ci);
            if (i + 1 < nr) face(c + 1, cf.co);
            if (k > 0) face(c - nr, cf.cz);
            else { b += 2.0 * cf.cz * v_lo; s += 2.0 * cf.cz * (v_lo - pc); }
            if (k + 1 < nz) face(c + nr, cf.cz);
            else { b += 2.0 * cf.cz * v_hi; s += 2.0 * cf.cz * (v_hi - pc); }
            r[c] = s;
            g0[c] = s;
            acc[0] += b * b;
            acc[1] += s * s;
        }
    }
    double tot[2];
    if (axi_sums<2>(acc, part, ctr, tot)) {
        sc[A_B2] = tot[0];
        sc[A_R2] = tot[1];
    }
}

// One colour of red-black Gauss-Seidel.  Thread (ii, k0) takes the cells
// 2 ii + ((k + colour) & 1) of ROWS planes; their loads come first (the
// other colour's values, not written here).
template <int ROWS> __global__ void __launch_bounds__(AX * AZ) k_axi_smooth(double* __restrict__ e, const double* __restrict__ g,
                                                        const uint8_t* __restrict__ m, const double* __restrict__ rd,
                                                        int nr, int nz, int color) {
    pdl_wait();
    const int ii = blockIdx.x * AX + threadIdx.x, k0 = (blockIdx.y * AZ + threadIdx.y) * ROWS;
    if (2 * ii >= nr) return;
    const double c0 = (double)(2 * ii);
    double xm[ROWS], xp[ROWS], zm[ROWS], zp[ROWS], gv[ROWS], rv[ROWS];
    bool ok[ROWS];
#pragma unroll
    for (int d = 0; d < ROWS; ++d) {
        const int k = k0 + d, par = (k + color) & 1, i = 2 * ii + par, c = k * nr + i;
        const bool in = k < nz && i < nr;
        ok[d] = in && !m[in ? c : 0];
        xm[d] = in && i > 0 ? e[c - 1] : 0.0;
        xp[d] = in && i + 1 < nr ? e[c + 1] : 0.0;
        zm[d] = in && k > 0 ? e[c - nr] : 0.0;
        zp[d] = in && k + 1 < nz ? e[c + nr] : 0.0;
        gv[d] = in ? g[c] : 0.0;
        rv[d] = in ? rd[(k == 0 || k == nz - 1 ? nr : 0) + i] : 0.0;
    }
#pragma unroll
    for (int d = 0; d < ROWS; ++d) {
        const int k = k0 + d, par = (k + color) & 1;
        const double ci = par ? c0 + 1.0 : c0;
        double s = ci * xm[d];
        s += (ci + 1.0) * xp[d];  // xp = 0 at the outer cylinder
        s += (ci + 0.5) * zm[d];
        s += (ci + 0.5) * zp[d];
        if (ok[d]) e[k * nr + 2 * ii + par] = (gv[d] + s) * rv[d];
    }
}

// The first full sweep from e = 0: red cells g rd, black cells from those of
// their neighbours (the x ones from the adjacent lanes where they hold them).
template <int ROWS> __global__ void __launch_bounds__(AX * AZ) k_axi_sweep_first(double* __restrict__ e, const double* __restrict__ g,
                                                             const uint8_t* __restrict__ m,
                                                             const double* __restrict__ rd, int nr, int nz) {
    pdl_wait();
    const int lane = threadIdx.x, ii = blockIdx.x * AX + lane, k0 = (blockIdx.y * AZ + threadIdx.y) * ROWS;
    auto red = [&](int i, int k) -> double {
        if (i < 0 || i >= nr || k < 0 || k >= nz) return 0.0;
        const int c = k * nr + i;
        return m[c] ? 0.0 : g[c] * rd[(k == 0 || k == nz - 1 ? nr : 0) + i];
    };
    const double c0 = (double)(2 * ii);
#pragma unroll
    for (int d = 0; d < ROWS; ++d) {
        const int k = k0 + d, par = k & 1, i0 = 2 * ii + par, i1 = 2 * ii + 1 - par;
        const double v0 = red(i0, k);
        const double prev = __shfl_up_sync(kFull, v0, 1), next = __shfl_down_sync(kFull, v0, 1);
        if (k >= nz) continue;
        if (i0 < nr) e[k * nr + i0] = v0;
        if (i1 >= nr) continue;
        double xm, xp;
        if (par) {  // i1 = 2 ii: its left neighbour is the previous pair's red cell
            xm = lane > 0 ? prev : red(i1 - 1, k);
            xp = v0;
        } else {
            xm = v0;
            xp = lane < AX - 1 ? next : red(i1 + 1, k);
        }
        const int c = k * nr + i1;
        const double ci = par ? c0 : c0 + 1.0;
        double s = ci * xm;
        s += i1 + 1 < nr ? (ci + 1.0) * xp : 0.0;
        s += (ci + 0.5) * red(i1, k - 1);
        s += (ci + 0.5) * red(i1, k + 1);
        e[c] = m[c] ? 0.0 : (g[c] + s) * rd[(k == 0 || k == nz - 1 ? nr : 0) + i1];
    }
}

// Half the sum of the children's residuals; the two black ones are zero (to
// rounding) after a black half-sweep, so the red ones are evaluated.
__global__ void __launch_bounds__(AX * AZ) k_axi_resid_restrict(const double* __restrict__ e,
                                                                const double* __restrict__ g,
                                                                const uint8_t* __restrict__ m, int nr, int nz,
                                                                double* __restrict__ gc,
                                                                const uint8_t* __restrict__ mc) {
    pdl_wait();
    const int cr = nr / 2, cz = nz / 2;
    const int I = blockIdx.x * AX + threadIdx.x, K = blockIdx.y * AZ + threadIdx.y;
    if (I >= cr || K >= cz) return;
    const int qc = K * cr + I;
    if (mc[qc]) { gc[qc] = 0.0; return; }
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        const int i = 2 * I + d, k = 2 * K + d, c = k * nr + i;
        const Coef cf = coef(i, nr);
        const double v = g[c] - (diag_of(cf, k, nz) * e[c] - nb_e(e, i, k, nr, nz, cf));
        acc += m[c] ? 0.0 : v;
    }
    gc[qc] = 0.5 * acc;
}

__device__ __forceinline__ double acval(const double* ec, int I, int K, int cr, int cz) {
    double sgn = 1.0;
    I = I < 0 ? 0 : (I >= cr ? cr - 1 : I);
    if (K < 0) { K = 0; sgn = -1.0; }
    if (K >= cz) { K = cz - 1; sgn = -1.0; }
    return sgn * ec[K * cr + I];
}

// The red cells take the bilinear interpolation of the coarser level's e; the
// black ones are formed anew by the half-sweep that follows, from red
// neighbours alone.  A thread takes both red cells of a coarse cell.
__global__ void __launch_bounds__(AX * AZ) k_axi_prolong_add(const double* __restrict__ ec, double* __restrict__ ef,
                                                             const uint8_t* __restrict__ m, int nr, int nz) {
    pdl_wait();
    const int cr = nr / 2, cz = nz / 2;
    const int I = blockIdx.x * AX + threadIdx.x, K = blockIdx.y * AZ + threadIdx.y;
    if (I >= cr || K >= cz) return;
    const double v = ec[K * cr + I];
#pragma unroll
    for (int d = 0; d < 2; ++d) {
        const int c = (2 * K + d) * nr + 2 * I + d, s = d ? 1 : -1;
        if (m[c]) continue;
        double acc = 0.5625 * v;
        acc += 0.1875 * acval(ec, I + s, K, cr, cz);
        acc += 0.1875 * acval(ec, I, K + s, cr, cz);
        acc += 0.0625 * acval(ec, I + s, K + s, cr, cz);
        ef[c] += acc;
    }
}

// Coarsest level that is too large for the one-block kernel: zero start and
// `sweeps` red-black sweeps in one block.
__global__ void __launch_bounds__(1024) k_axi_coarse(double* e, const double* g, const uint8_t* m,
                                                     const double* __restrict__ rd, int nr, int nz, int sweeps) {
    pdl_wait();
    const int n = nr * nz;
    for (int c = threadIdx.x; c < n; c += blockDim.x) e[c] = 0.0;
    __syncthreads();
    for (int s = 0; s < 2 * sweeps; ++s) {
        const int color = s & 1;
        for (int c = threadIdx.x; c < n; c += blockDim.x) {
            const int i = c % nr, k = c / nr;
            if (((i + k) & 1) != color || m[c]) continue;
            const Coef cf = coef(i, nr);
            e[c] = (g[c] + nb_e(e, i, k, nr, nz, cf)) * rd[(k == 0 || k == nz - 1 ? nr : 0) + i];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- small levels
// Levels of at most kATailCells cells in one block, as poisson_tail.cuh: a
// thread owns one cell of each colour of a level, e stands in shared memory
// with an array per colour.  The coarsest level's sweeps end as soon as one
// changes nothing (the rest would not either).  Double operations of one
// multiprocessor bound it above 32 x 32 (16 warps x 7 operations x 18 clocks
// a half-sweep), so larger levels are kernels of their own.
constexpr int kATailLevels = 8, kATailCells = 1024;
struct AxiTailLevel {
    int nr, nz, hr, h, ca, act;
    int e, r, g;  // shared memory, doubles: e of both colours, residuals, g of both colours
    const uint8_t* m;
    const double* rd;
};
struct AxiTail {
    AxiTailLevel L[kATailLevels];
    double* e_first;
    const double* g_first;
    int levels, words, pre, post, coarse;
};
inline AxiTailLevel axi_tail_geometry(int nr, int nz) {
    AxiTailLevel L = {};
    L.nr = nr;
    L.nz = nz;
    L.hr = (nr + 1) / 2;
    L.h = nz * L.hr;
    L.ca = (nz + 2) * L.hr;
    L.act = (L.h + 31) & ~31;
    return L;
}

struct AxiCell {
    double g, rd, ci, co, cz;
    int o, b;  // places of the cell and of its right neighbour's slot, each in its colour's array
    int i, k;
    bool xm, xp, in, on;  // neighbours in r exist; the cell exists; and is not held at zero
};
__device__ __forceinline__ AxiCell axi_cell(const AxiTailLevel& L, int t, int color) {
    AxiCell c;
    const int tt = t < L.h ? t : 0, ii = tt % L.hr;
    c.k = tt / L.hr;
    c.i = 2 * ii + ((c.k + color) & 1);
    c.in = t < L.h && c.i < L.nr;
    c.on = c.in && !L.m[c.in ? c.k * L.nr + c.i : 0];
    c.o = (c.k + 1) * L.hr + ii;
    c.b = c.o + ((c.k + color) & 1);
    c.xm = c.i > 0;
    c.xp = c.i + 1 < L.nr;
    c.ci = (double)c.i;
    c.cz = c.ci + 0.5;
    c.co = c.xp ? c.ci + 1.0 : 0.0;
    c.rd = c.on ? L.rd[(c.k == 0 || c.k == L.nz - 1 ? L.nr : 0) + c.i] : 0.0;
    c.g = 0.0;
    return c;
}
__device__ __forceinline__ double axi_sum(const AxiCell& c, int hr, const double* en) {
    double s = c.ci * (c.xm ? en[c.b - 1] : 0.0);
    s += c.co * (c.xp ? en[c.b] : 0.0);
    s += c.cz * en[c.o - hr];
    s += c.cz * en[c.o + hr];
    return s;
}
// Sweeps of a level: n times red, black, or (black_first) black, red; with
// `settle` (a level of one warp) until a sweep changes nothing.
__device__ __forceinline__ void axi_sweeps(const AxiTailLevel& L, const AxiCell (&c)[2], double* e, int n, bool black_first,
                                           bool settle, int id) {
    const int turns = black_first ? n + 1 : n;
#pragma unroll 1
    for (int s = 0; s < turns; ++s) {
        bool changed = false;
        if (!black_first || s > 0) {
            const double v = (c[0].g + axi_sum(c[0], L.hr, e + L.ca)) * c[0].rd;
            if (c[0].on) {
                changed |= settle && e[c[0].o] != v;
                e[c[0].o] = v;
            }
            bar_named(id, L.act);
        }
        if (!black_first || s < n) {
            const double v = (c[1].g + axi_sum(c[1], L.hr, e)) * c[1].rd;
            if (c[1].on) {
                changed |= settle && e[L.ca + c[1].o] != v;
                e[L.ca + c[1].o] = v;
            }
            bar_named(id, L.act);
        }
        if (settle && !__any_sync(kFull, changed)) break;
    }
}

__global__ void __launch_bounds__(512, 1) k_axi_tail(const __grid_constant__ AxiTail T) {
    extern __shared__ __align__(16) double axi_sm[];
    const int t = threadIdx.x, last = T.levels - 1;
    for (int p = t; p < T.words; p += blockDim.x) axi_sm[p] = 0.0;
    pdl_wait();
    __syncthreads();
    int l = 0;
#pragma unroll 1
    for (; l <= last; ++l) {
        const AxiTailLevel L = T.L[l];
        if (t >= L.act) break;
        AxiCell c[2] = {axi_cell(L, t, 0), axi_cell(L, t, 1)};
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (l == 0) {
                if (c[q].in) c[q].g = T.g_first[c[q].k * L.nr + c[q].i];
            } else if (c[q].on) {
                const AxiTailLevel& F = T.L[l - 1];
                const double* R = axi_sm + F.r;
                c[q].g = 0.5 * (R[2 * c[q].k * F.hr + c[q].i] + R[(2 * c[q].k + 1) * F.hr + c[q].i]);
            }
            if (t < L.h) axi_sm[L.g + q * L.h + t] = c[q].g;
        }
        double* e = axi_sm + L.e;
        axi_sweeps(L, c, e, l == last ? T.coarse : T.pre, false, l == last && L.act == 32, l + 1);
        if (l < last) {
            const double d = c[0].ci + c[0].co + 2.0 * c[0].cz + (c[0].k == 0 ? c[0].cz : 0.0) +
                             (c[0].k == L.nz - 1 ? c[0].cz : 0.0);
            const double v = c[0].g - (d * e[c[0].o] - axi_sum(c[0], L.hr, e + L.ca));
            if (t < L.h) axi_sm[L.r + t] = c[0].on ? v : 0.0;
            bar_named(l + 1, L.act);
        }
    }
#pragma unroll 1
    for (--l; l >= 0; --l) {
        if (l == last) continue;
        const AxiTailLevel L = T.L[l];
        bar_named(l + 1, L.act);  // the coarser level is done
        const AxiTailLevel& D = T.L[l + 1];
        AxiCell c[2] = {axi_cell(L, t, 0), axi_cell(L, t, 1)};
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (t < L.h) c[q].g = axi_sm[L.g + q * L.h + t];
        double* e = axi_sm + L.e;
        if (c[0].on) {
            const double* ec = axi_sm + D.e;
            auto at = [&](int I, int K) -> double {
                double sgn = 1.0;
                I = I < 0 ? 0 : (I >= D.nr ? D.nr - 1 : I);
                if (K < 0) { K = 0; sgn = -1.0; }
                if (K >= D.nz) { K = D.nz - 1; sgn = -1.0; }
                return sgn * ec[((I + K) & 1) * D.ca + (K + 1) * D.hr + (I >> 1)];
            };
            const int I = c[0].i >> 1, K = c[0].k >> 1, si = (c[0].i & 1) ? 1 : -1, sk = (c[0].k & 1) ? 1 : -1;
            double acc = 0.5625 * at(I, K);
            acc += 0.1875 * at(I + si, K);
            acc += 0.1875 * at(I, K + sk);
            acc += 0.0625 * at(I + si, K + sk);
            e[c[0].o] += acc;
        }
        bar_named(l + 1, L.act);
        axi_sweeps(L, c, e, T.post, true, false, l + 1);
    }
    __syncthreads();
    const AxiTailLevel& L0 = T.L[0];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const AxiCell c = axi_cell(L0, t, q);
        if (c.in) T.e_first[c.k * L0.nr + c.i] = axi_sm[L0.e + q * L0.ca + c.o];
    }
}

// ---------------------------------------------------------------- CG iteration
// Two kernels, as in the float32 Cartesian solve: w = A z with the sums z.r,
// z.q_prev and z.w, from which the last block forms beta, gamma = p.q (A is
// symmetric) and alpha; then p = z + beta p, q = w + beta q, phi += alpha p,
// r -= alpha q and ||r||^2.
__global__ void __launch_bounds__(AX * AZ) k_axi_apply(const double* __restrict__ z, const double* __restrict__ r,
                                                       const double* __restrict__ q, const uint8_t* __restrict__ m, int nr,
                                                       int nz, double* __restrict__ w, int first, double* part,
                                                       unsigned* ctr, double* sc) {
    pdl_wait();
    const int i = blockIdx.x * AX + threadIdx.x, k0 = (blockIdx.y * AZ + threadIdx.y) * kRows;
    double acc[3] = {0.0, 0.0, 0.0};
    if (i < nr) {
        const Coef cf = coef(i, nr);
        const double din = cf.ci + cf.co + 2.0 * cf.cz;
        double col[kRows + 2], xm[kRows], xp[kRows], rv[kRows], qv[kRows];
#pragma unroll
        for (int d = 0; d < kRows + 2; ++d) {
            const int k = k0 - 1 + d;
            col[d] = k >= 0 && k < nz ? z[k * nr + i] : 0.0;
        }
#pragma unroll
        for (int d = 0; d < kRows; ++d) {
            const int k = k0 + d, c = k * nr + i;
            const bool in = k < nz;
            xm[d] = in && i > 0 ? z[c - 1] : 0.0;
            xp[d] = in && i + 1 < nr ? z[c + 1] : 0.0;
            rv[d] = in ? r[c] : 0.0;
            qv[d] = in && !first ? q[c] : 0.0;
        }
#pragma unroll
        for (int d = 0; d < kRows; ++d) {
            const int k = k0 + d, c = k * nr + i;
            if (k >= nz) break;
            double s = cf.ci * xm[d];
            s += cf.co * xp[d];
            s += cf.cz * col[d];
            s += cf.cz * col[d + 2];
            const double diag = k == 0 || k == nz - 1 ? din + cf.cz : din;
            const double v = m[c] ? 0.0 : diag * col[d + 1] - s;
            w[c] = v;
            acc[0] += col[d + 1] * rv[d];
            if (!first) acc[1] += col[d + 1] * qv[d];
            acc[2] += col[d + 1] * v;
        }
    }
    double tot[3];
    if (axi_sums<3>(acc, part, ctr, tot)) {
        const double rho_old = sc[A_RHO];
        const double beta = first || rho_old == 0.0 ? 0.0 : -sc[A_ALPHA] * tot[1] / rho_old;
        const double gam = first ? tot[2] : tot[2] + beta * (2.0 * tot[1] + beta * sc[A_GAM]);
        sc[A_BETA] = beta;
        sc[A_RHO] = tot[0];
        sc[A_GAM] = gam;
        sc[A_ALPHA] = gam > 0.0 ? tot[0] / gam : 0.0;
    }
}

__global__ void __launch_bounds__(AX * AZ) k_axi_step(const double* __restrict__ z, const double* __restrict__ w,
                                                      double* __restrict__ p, double* __restrict__ q,
                                                      double* __restrict__ phi, double* __restrict__ r,
                                                      double* __restrict__ g0, int n, int first, double* part,
                                                      unsigned* ctr, double* sc) {
    pdl_wait();
    const double a = sc[A_ALPHA], b = first ? 0.0 : sc[A_BETA];
    double acc[1] = {0.0};
    const int stride = gridDim.x * AX * AZ;
    for (int c = blockIdx.x * AX * AZ + threadIdx.y * AX + threadIdx.x; c < n; c += stride) {
        double pp = z[c], qq = w[c];
        if (b != 0.0) {
            pp += b * p[c];
            qq += b * q[c];
        }
        p[c] = pp;
        q[c] = qq;
        phi[c] += a * pp;
        const double rr = r[c] - a * qq;
        r[c] = rr;
        g0[c] = rr;
        acc[0] += rr * rr;
    }
    double tot[1];
    if (axi_sums<1>(acc, part, ctr, tot)) sc[A_R2] = tot[0];
}

template <class T>
__global__ void __launch_bounds__(AX * AZ) k_axi_grad(const double* __restrict__ phi, int nr, int nz, double h, double v_lo,
                                                      double v_hi, float* Er, float* Ez, T* E4) {
    ACELL
    if (!in) return;
    const double inv = 1.0 / (2.0 * h), pc = phi[c];
    const double rm = i > 0 ? phi[c - 1] : pc, rp = i + 1 < nr ? phi[c + 1] : pc;
    const double zm = k > 0 ? phi[c - nr] : 2.0 * v_lo - pc, zp = k + 1 < nz ? phi[c + nr] : 2.0 * v_hi - pc;
    const double er = -(rp - rm) * inv, ez = -(zp - zm) * inv;
    if (Er) { Er[c] = (float)er; Ez[c] = (float)ez; }
    if (E4) {
        if (sizeof(T) == 4) {
            reinterpret_cast<float4*>(E4)[c] = make_float4((float)er, 0.0f, (float)ez, 0.0f);
        } else {
            E4[4 * c] = (T)er; E4[4 * c + 1] = (T)0; E4[4 * c + 2] = (T)ez; E4[4 * c + 3] = (T)0;
        }
    }
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr unsigned kStepBlocks = 608;  // of the update kernel at most
dim3 grid_step(int n) {
    const unsigned b = (unsigned)((n + AX * AZ - 1) / (AX * AZ));
    return dim3(b < kStepBlocks ? b : kStepBlocks);
}

}  // namespace

void AxiMG::plan(int nr, int nz) {
    levels = 0;
    int a = nr, b = nz;
    for (;;) {
        lr[levels] = a;
        lz[levels] = b;
        ++levels;
        if (levels >= kMaxLevels || (a % 2) || (b % 2) || a < 4 || b < 4) break;
        a /= 2;
        b /= 2;
    }
}

bool AxiMG::supported(int nr, int nz) {
    if (nr < 2 || nz < 2 || (long long)nr * nz > 0x7fffffffLL) return false;
    AxiMG g;
    g.plan(nr, nz);
    return (long long)g.lr[g.levels - 1] * g.lz[g.levels - 1] <= 4096;
}

size_t AxiMG::bytes(int nr, int nz) {
    AxiMG g;
    return g.carve(nullptr, nr, nz);
}

size_t AxiMG::carve(void* base, int nr, int nz) {
    plan(nr, nz);
    uintptr_t pp = (uintptr_t)base;
    const uintptr_t p0 = pp;
    auto take = [&](size_t b) {
        void* o = (void*)pp;
        pp += al256(b);
        return o;
    };
    const size_t n0 = (size_t)nr * nz;
    norms = (double*)take(A_N * 8);
    loop = (AxiLoop*)take(sizeof(AxiLoop));
    ctr = (unsigned*)take(4 * sizeof(unsigned));
    const dim3 gr = agrid_rows(nr, nz);
    const size_t blocks = (size_t)gr.x * gr.y > kStepBlocks ? (size_t)gr.x * gr.y : kStepBlocks;
    part = (double*)take(blocks * 3 * 8);
    r = (double*)take(n0 * 8);
    p = (double*)take(n0 * 8);
    q = (double*)take(n0 * 8);
    w = (double*)take(n0 * 8);
    for (int l = 0; l < levels; ++l) {
        const size_t n = (size_t)lr[l] * lz[l];
        e[l] = (double*)take(n * 8);
        g[l] = (double*)take(n * 8);
        m[l] = (uint8_t*)take(n);
        rd[l] = (double*)take((size_t)2 * lr[l] * 8);
    }
    return (size_t)(pp - p0);
}

cudaError_t AxiMG::build_masks(const uint8_t* mask, cudaStream_t s) {
    const int n0 = lr[0] * lz[0];
    k_axi_copy_mask<<<(n0 + 255) / 256, 256, 0, s>>>(mask, m[0], n0);
    for (int l = 1; l < levels; ++l)
        k_axi_restrict_mask<<<agrid(lr[l], lz[l]), kABlk, 0, s>>>(m[l - 1], lr[l - 1], lz[l - 1], m[l]);
    for (int l = 0; l < levels; ++l) k_axi_rdiag<<<(lr[l] + 127) / 128, 128, 0, s>>>(lr[l], lz[l], rd[l]);
    launches += 2 * levels;
    return cudaGetLastError();
}

// First level of the one-block kernel: at most kATailCells cells and
// kATailLevels levels from there; `levels` when the coarsest is larger.
int AxiMG::tail_level() const {
    for (int l = 0; l < levels; ++l)
        if (lr[l] * lz[l] <= kATailCells && lz[l] * ((lr[l] + 1) / 2) <= 512 && levels - l <= kATailLevels) return l;
    return levels;
}

// One V(pre, post)-cycle on A e0 = g0; e0 is overwritten.
void AxiMG::vcycle(cudaStream_t s) {
    const int tl = tail_level(), top = tl < levels ? tl : levels - 1;
    for (int l = 0; l < top; ++l) {
        note(launch_pdl(deep(lr[l], lz[l]) ? k_axi_sweep_first<kRows> : k_axi_sweep_first<1>, agrid_half(lr[l], lz[l]),
                        kABlk, 0, s, e[l], (const double*)g[l], (const uint8_t*)m[l], (const double*)rd[l], lr[l], lz[l]));
        for (int it = 1; it < pre; ++it)
            for (int col = 0; col < 2; ++col)
                note(launch_pdl(deep(lr[l], lz[l]) ? k_axi_smooth<kRows> : k_axi_smooth<1>, agrid_half(lr[l], lz[l]), kABlk,
                                0, s, e[l], (const double*)g[l], (const uint8_t*)m[l], (const double*)rd[l], lr[l], lz[l],
                                col));
        note(launch_pdl(k_axi_resid_restrict, agrid(lr[l + 1], lz[l + 1]), kABlk, 0, s, (const double*)e[l],
                        (const double*)g[l], (const uint8_t*)m[l], lr[l], lz[l], g[l + 1], (const uint8_t*)m[l + 1]));
    }
    if (tl < levels) {
        AxiTail T = {};
        for (int l = tl; l < levels; ++l) {
            AxiTailLevel& L = T.L[T.levels++];
            L = axi_tail_geometry(lr[l], lz[l]);
            L.m = m[l];
            L.rd = rd[l];
            L.e = T.words;
            L.r = L.e + 2 * L.ca;
            L.g = L.r + L.h;
            T.words = L.g + 2 * L.h;
        }
        T.e_first = e[tl];
        T.g_first = g[tl];
        T.pre = pre;
        T.post = post;
        T.coarse = coarse_sweeps;
        // at most 31 KB (256 x 4 cells): no opt-in needed
        note(launch_pdl(k_axi_tail, dim3(1), dim3(T.L[0].act), (size_t)T.words * 8, s, T));
    } else {
        note(launch_pdl(k_axi_coarse, dim3(1), dim3(1024), 0, s, e[top], (const double*)g[top], (const uint8_t*)m[top],
                        (const double*)rd[top], lr[top], lz[top], coarse_sweeps));
    }
    for (int l = top - 1; l >= 0; --l) {
        note(launch_pdl(k_axi_prolong_add, agrid(lr[l + 1], lz[l + 1]), kABlk, 0, s, (const double*)e[l + 1], e[l],
                        (const uint8_t*)m[l], lr[l], lz[l]));
        for (int it = 0; it < post; ++it)
            for (int col = 1; col >= 0; --col)
                note(launch_pdl(deep(lr[l], lz[l]) ? k_axi_smooth<kRows> : k_axi_smooth<1>, agrid_half(lr[l], lz[l]), kABlk,
                                0, s, e[l], (const double*)g[l], (const uint8_t*)m[l], (const double*)rd[l], lr[l], lz[l],
                                col));
    }
    launches += (long long)top * (2 * pre - 1 + 2 * post + 2) + 1;
}

void AxiMG::iteration(cudaStream_t s, double* phi, bool first) {
    const int nr = lr[0], nz = lz[0], n = nr * nz, f = first ? 1 : 0;
    vcycle(s);
    note(launch_pdl(k_axi_apply, agrid_rows(nr, nz), kABlk, 0, s, (const double*)e[0], (const double*)r, (const double*)q,
                    (const uint8_t*)m[0], nr, nz, w, f, part, ctr + 1, norms));
    note(launch_pdl(k_axi_step, grid_step(n), kABlk, 0, s, (const double*)e[0], (const double*)w, p, q, phi, r, g[0], n,
                    f, part, ctr + 2, norms));
    launches += 2;
}

namespace {
void launch_resid(const AxiMG& a, cudaStream_t s, double* phi, const AxiCharge& rho, double h, double v_lo, double v_hi,
                  double v_mask) {
    const int nr = a.lr[0], nz = a.lz[0];
    const double h2e = h * h / kEps0;
    if (rho.rho)
        k_axi_resid<false><<<agrid_rows(nr, nz), kABlk, 0, s>>>(phi, rho, a.m[0], nr, nz, h2e, v_lo, v_hi, v_mask, a.r,
                                                                a.g[0], a.part, a.ctr, a.norms);
    else
        k_axi_resid<true><<<agrid_rows(nr, nz), kABlk, 0, s>>>(phi, rho, a.m[0], nr, nz, h2e, v_lo, v_hi, v_mask, a.r,
                                                               a.g[0], a.part, a.ctr, a.norms);
}
}  // namespace

int AxiMG::solve(const AxiCharge& rho, const uint8_t* mask, double* phi, double h, double v_lo, double v_hi,
                 double v_mask, double rtol, int max_cycles, int packed_prec, void* E4, float* Er, float* Ez,
                 cudaStream_t s, int* cycles_out, double* rel_out, double* host_norms) {
    launch_err = cudaSuccess;
    const int nr = lr[0], nz = lz[0];
    if (!persistent || !masks_ready) {
        if (build_masks(mask, s) != cudaSuccess) return PIC_ERR_CUDA;
        masks_ready = true;
    }
    cudaMemsetAsync(ctr, 0, 4 * sizeof(unsigned), s);
    launch_resid(*this, s, phi, rho, h, v_lo, v_hi, v_mask);
    ++launches;
    int cyc = 0, rc = PIC_OK;
    double bn = 1.0, rn = 0.0;
    for (;;) {
        if (cudaMemcpyAsync(host_norms, norms, 2 * 8, cudaMemcpyDeviceToHost, s) != cudaSuccess) return PIC_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return PIC_ERR_CUDA;
        bn = host_norms[A_B2] > 0.0 ? sqrt(host_norms[A_B2]) : 1.0;
        rn = sqrt(host_norms[A_R2]);
        if (rn / bn <= rtol) break;
        if (cyc >= max_cycles) { rc = PIC_ERR_TIMEOUT; break; }
        iteration(s, phi, cyc == 0);
        if (!launched()) return PIC_ERR_CUDA;
        ++cyc;
    }
    if (cycles_out) *cycles_out = cyc;
    if (rel_out) *rel_out = rn / bn;
    if (E4 || Er) {
        if (packed_prec == 64)
            k_axi_grad<double><<<agrid(nr, nz), kABlk, 0, s>>>(phi, nr, nz, h, v_lo, v_hi, Er, Ez, (double*)E4);
        else
            k_axi_grad<float><<<agrid(nr, nz), kABlk, 0, s>>>(phi, nr, nz, h, v_lo, v_hi, Er, Ez, (float*)E4);
        ++launches;
    }
    return cudaGetLastError() == cudaSuccess ? rc : PIC_ERR_CUDA;
}

// Decisions of a device-driven solve, as the host loop takes them: no further
// iteration when ||r|| / ||b|| <= rtol or the cycle limit is reached
// (flagged).
__device__ __forceinline__ bool axi_go(const double* sc, AxiLoop* L, double rtol, int max_cycles) {
    const double bn = sc[A_B2] > 0.0 ? sqrt(sc[A_B2]) : 1.0;
    const double rn = sqrt(sc[A_R2]);
    L->rel = rn / bn;
    ++L->trips;
    if (rn / bn <= rtol) return false;
    if (L->cyc >= max_cycles) {
        L->timeout = 1;
        return false;
    }
    return true;
}
// Before the first iteration (branch 0) and before the loop over the later
// ones (branch 1): the condition of the if node that holds them.
__global__ void k_axi_decide(const double* __restrict__ sc, AxiLoop* L, double rtol, int max_cycles, int branch,
                             cudaGraphConditionalHandle h) {
    const bool go = axi_go(sc, L, rtol, max_cycles);
    if (go && branch == 0) {
        L->cyc = 1;
        L->n_branch[0] = 1;
    }
    cudaGraphSetConditional(h, go ? 1u : 0u);
}
// After a later iteration: counts it and sets the loop's condition (every trip
// counts, so the cycle limit ends the loop).
__global__ void k_axi_trip(const double* __restrict__ sc, AxiLoop* L, double rtol, int max_cycles,
                           cudaGraphConditionalHandle h_loop) {
    ++L->cyc;
    ++L->n_branch[1];
    cudaGraphSetConditional(h_loop, axi_go(sc, L, rtol, max_cycles) ? 1u : 0u);
}

__global__ void k_axi_report(const AxiLoop* __restrict__ L, int* cycles, double* rel, unsigned* err, unsigned bit,
                             unsigned long long* kernels, int kb0, int kb1) {
    *cycles = L->cyc;
    *rel = L->rel;
    if (L->timeout) *err |= bit;
    *kernels += (unsigned long long)L->trips + (unsigned long long)L->n_branch[0] * kb0 +
                (unsigned long long)L->n_branch[1] * kb1;
}

int AxiMG::prepare_capture() {
    for (int q = 0; q < 3; ++q)
        if (!cap_body[q] && cudaStreamCreateWithFlags(&cap_body[q], cudaStreamNonBlocking) != cudaSuccess)
            return PIC_ERR_CUDA;
    return PIC_OK;
}

void AxiMG::release() {
    for (int q = 0; q < 3; ++q)
        if (cap_body[q]) { cudaStreamDestroy(cap_body[q]); cap_body[q] = nullptr; }
}

// The loop over the later iterations: the decision after an iteration sets
// the loop's condition, so a trip is an iteration and its decision.
int AxiMG::capture_solve(cudaStream_t cs, const AxiCharge& rho, double* phi, double h, double v_lo, double v_hi,
                         double v_mask, double rtol, int max_cycles, int packed_prec, void* E4, int* cycles_dst,
                         double* rel_dst, unsigned* err_dst, unsigned err_bit, unsigned long long* kernels_dst,
                         long long* fixed_kernels) {
    if (!loop || !masks_ready || !cap_body[0] || !cap_body[1] || !cap_body[2]) return PIC_ERR_STATE;
    launch_err = cudaSuccess;
    const int nr = lr[0], nz = lz[0];
    cudaGraph_t top = capturing_graph(cs), first = nullptr, more = nullptr, body = nullptr;
    if (!top) return PIC_ERR_CUDA;
    cudaMemsetAsync(ctr, 0, 4 * sizeof(unsigned), cs);
    cudaMemsetAsync(loop, 0, sizeof(AxiLoop), cs);
    launch_resid(*this, cs, phi, rho, h, v_lo, v_hi, v_mask);
    const auto capture_into = [](cudaStream_t s, cudaGraph_t g) {
        return cudaStreamBeginCaptureToGraph(s, g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    };
    cudaGraphConditionalHandle h_first, h_more, h_loop;
    if (cudaGraphConditionalHandleCreate(&h_first, top, 0u, cudaGraphCondAssignDefault) != cudaSuccess) return PIC_ERR_CUDA;
    k_axi_decide<<<1, 1, 0, cs>>>(norms, loop, rtol, max_cycles, 0, h_first);
    if (add_conditional(cs, h_first, cudaGraphCondTypeIf, 1, &first) != cudaSuccess) return PIC_ERR_CUDA;
    int kb[2];
    const long long l0 = launches;
    // the first iteration, then the loop only if it did not reach the tolerance
    if (capture_into(cap_body[0], first) != cudaSuccess) return PIC_ERR_CUDA;
    iteration(cap_body[0], phi, true);
    kb[0] = (int)(launches - l0);
    bool ok = cudaGraphConditionalHandleCreate(&h_more, first, 0u, cudaGraphCondAssignDefault) == cudaSuccess;
    if (ok) {
        k_axi_decide<<<1, 1, 0, cap_body[0]>>>(norms, loop, rtol, max_cycles, 1, h_more);
        ok = add_conditional(cap_body[0], h_more, cudaGraphCondTypeIf, 1, &more) == cudaSuccess;
    }
    ok = end_body_capture(cap_body[0]) == cudaSuccess && ok;
    if (!ok) return PIC_ERR_CUDA;
    if (cudaGraphConditionalHandleCreate(&h_loop, more, 1u, cudaGraphCondAssignDefault) != cudaSuccess) return PIC_ERR_CUDA;
    if (capture_into(cap_body[1], more) != cudaSuccess) return PIC_ERR_CUDA;
    ok = add_conditional(cap_body[1], h_loop, cudaGraphCondTypeWhile, 1, &body) == cudaSuccess;
    ok = end_body_capture(cap_body[1]) == cudaSuccess && ok;
    if (!ok) return PIC_ERR_CUDA;
    if (capture_into(cap_body[2], body) != cudaSuccess) return PIC_ERR_CUDA;
    const long long l1 = launches;
    iteration(cap_body[2], phi, false);
    kb[1] = (int)(launches - l1);
    k_axi_trip<<<1, 1, 0, cap_body[2]>>>(norms, loop, rtol, max_cycles, h_loop);
    if (end_body_capture(cap_body[2]) != cudaSuccess) return PIC_ERR_CUDA;
    long long fixed = 2;  // residual, report
    if (E4) {
        if (packed_prec == 64)
            k_axi_grad<double><<<agrid(nr, nz), kABlk, 0, cs>>>(phi, nr, nz, h, v_lo, v_hi, nullptr, nullptr,
                                                                 (double*)E4);
        else
            k_axi_grad<float><<<agrid(nr, nz), kABlk, 0, cs>>>(phi, nr, nz, h, v_lo, v_hi, nullptr, nullptr,
                                                                (float*)E4);
        ++fixed;
    }
    k_axi_report<<<1, 1, 0, cs>>>(loop, cycles_dst, rel_dst, err_dst, err_bit, kernels_dst, kb[0], kb[1]);
    if (fixed_kernels) *fixed_kernels = fixed;
    return launched() && cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

}  // namespace pic

using pic::AxiMG;

extern "C" size_t poisson_axi_workspace_bytes(int nr, int nz) {
    if (!AxiMG::supported(nr, nz)) return 0;
    return AxiMG::bytes(nr, nz);
}

extern "C" int poisson_axi_solve(int nr, int nz, double dx, double v_lo, double v_hi, double v_mask,
                                 const double* rho, const uint8_t* mask, double* phi, float* Er, float* Ez,
                                 double rtol, int max_cycles, void* ws, size_t ws_bytes, poisson_stats* st,
                                 pic_stream_t stream) {
    if (!rho || !phi || !ws || !(dx > 0) || !(rtol > 0) || max_cycles < 0 || !AxiMG::supported(nr, nz))
        return PIC_ERR_ARG;
    if ((Er == nullptr) != (Ez == nullptr)) return PIC_ERR_ARG;
    if (ws_bytes < AxiMG::bytes(nr, nz) || ((uintptr_t)ws & 255)) return PIC_ERR_ARG;
    AxiMG mg;
    mg.carve(ws, nr, nz);
    double hn[2];
    int cycles = 0;
    double rel = 0.0;
    const pic::AxiCharge charge{rho, nullptr, nullptr, nullptr, 0.0};
    const int rc = mg.solve(charge, mask, phi, dx, v_lo, v_hi, v_mask, rtol, max_cycles, 32, nullptr, Er, Ez,
                            (cudaStream_t)stream, &cycles, &rel, hn);
    if (st) { st->cycles = cycles; st->rel_res = rel; }
    return rc;
}

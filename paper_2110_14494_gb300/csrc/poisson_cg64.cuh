// Float64 flexible CG of the Cartesian solve (included by poisson.cu inside its
// anonymous namespace): the residual of the potential and the two kernels of
// an iteration, built as the float32 ones (poisson_mixed.cuh).  Threads walk
// ZC planes with their loads issued first; sums are per-block partials added
// in a fixed order by the last block.
//
// What bounds them: the double pipe (18 clocks of a multiprocessor for a warp's
// operation: a float's conversion, an addition, a product alike), so x
// neighbours come converted from the adjacent lanes, and the sums cost a block
// 24 warp operations a quantity instead of 60.  On 64 x 48 x 80 cells, before
// (blocks looping over planes with a dependent round trip each, six kernels an
// iteration) and now: residual and right-hand side 37.6 and 15 us, iteration
// without its V-cycle 45 and 25 us.
//
// q and p.q follow from recurrences (q = A z + beta q, poisson_mixed.cuh's
// cg_scalars) instead of A p.  The reported residual stays the true one as far
// as with A p formed each time: on grids from 16^3 to 128^3, random and smooth
// charges, both take the same iterations down to 1e-15; it equals the residual
// of the returned potential to 1 % at 1e-13, to a sixth at 1e-14, and below that
// the potential's own rounding (1e-15 to 6e-15) remains.

// Sums NV per-thread values over the grid, as grid_sums, in fewer double
// operations: warp q sums quantity q of its block, each lane four threads'
// values first.  Returns true in thread 0 of the last block, with the totals.
template <int NV> __device__ bool grid_sums64(const double (&v)[NV], double* part, unsigned* ctr, double (&tot)[NV]) {
    static_assert(NV <= BY, "a warp for each quantity");
    __shared__ double red[NV][BX * BY];
    __shared__ int last;
    const int t = threadIdx.x + threadIdx.y * BX, lane = t & 31, w = t >> 5;
    const unsigned b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
#pragma unroll
    for (int q = 0; q < NV; ++q) red[q][t] = v[q];
    __syncthreads();
    if (w < NV) {
        double s = (red[w][lane] + red[w][lane + 32]) + (red[w][lane + 64] + red[w][lane + 96]);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (lane == 0) {
            part[(size_t)b * NV + w] = s;
            __threadfence();
        }
    }
    __syncthreads();
    if (t == 0) last = atomicAdd(ctr, 1u) == nb - 1 ? 1 : 0;
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double s = 0.0;
        for (unsigned x0 = t; x0 < nb; x0 += 4u * BX * BY) {
            double a[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned x = x0 + u * BX * BY;
                a[u] = x < nb ? __ldcg(part + (size_t)x * NV + q) : 0.0;
            }
            s += a[0];
#pragma unroll
            for (int u = 1; u < 4; ++u)
                if (x0 + u * BX * BY < nb) s += a[u];
        }
        red[q][t] = s;
    }
    __syncthreads();
    if (w < NV) {
        double s = (red[w][lane] + red[w][lane + 32]) + (red[w][lane + 64] + red[w][lane + 96]);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
        if (lane == 0) red[w][0] = s;
    }
    __syncthreads();
    if (t != 0) return false;
#pragma unroll
    for (int q = 0; q < NV; ++q) tot[q] = red[q][0];
    *ctr = 0u;
    return true;
}

// r = b - A phi with the true boundary values and its float32 copy for the
// preconditioner; ||b||^2 with b = h^2 rho / eps0 + plate and electrode terms,
// ||r||^2; electrode cells get phi = v_mask (their neighbours use v_mask, not
// the value they may still hold).
// MANY: the block walks several slabs of planes (grid_cg64).
template <bool MANY>
__global__ void __launch_bounds__(BX * BY) k_resid64(double* __restrict__ phi, const double* __restrict__ rho,
                                                     const uint8_t* __restrict__ mask, int nx, int ny, int nz, double h2e,
                                                     double v_lo, double v_hi, double v_mask, double* __restrict__ r,
                                                     float* __restrict__ g0, double* part, unsigned* ctr, double* sc) {
    const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y;
    const bool in = i < nx && j < ny;
    const int pl = nx * ny, c0 = in ? lin(i, j, 0, nx, ny) : 0;
    double acc[2] = {0.0, 0.0};
    int k0 = blockIdx.z * ZC;
    if (in) do {
        double col[ZC + 2], xm[ZC], xp[ZC], ym[ZC], yp[ZC], rh[ZC];
        uint8_t cm[ZC + 2], mx[ZC], mp[ZC], my[ZC], mq[ZC];
#pragma unroll
        for (int d = 0; d < ZC + 2; ++d) {
            const int k = k0 - 1 + d;
            const bool ok = k >= 0 && k < nz;
            col[d] = ok ? phi[c0 + k * pl] : 0.0;
            cm[d] = ok ? mask[c0 + k * pl] : 0;
        }
#pragma unroll
        for (int d = 0; d < ZC; ++d) {
            const int k = k0 + d, c = c0 + k * pl;
            const bool ok = k < nz;
            xm[d] = ok && i > 0 ? phi[c - 1] : 0.0;
            mx[d] = ok && i > 0 ? mask[c - 1] : 0;
            xp[d] = ok && i < nx - 1 ? phi[c + 1] : 0.0;
            mp[d] = ok && i < nx - 1 ? mask[c + 1] : 0;
            ym[d] = ok && j > 0 ? phi[c - nx] : 0.0;
            my[d] = ok && j > 0 ? mask[c - nx] : 0;
            yp[d] = ok && j < ny - 1 ? phi[c + nx] : 0.0;
            mq[d] = ok && j < ny - 1 ? mask[c + nx] : 0;
            rh[d] = ok ? rho[c] : 0.0;
        }
#pragma unroll
        for (int d = 0; d < ZC; ++d) {
            const int k = k0 + d, c = c0 + k * pl;
            if (k >= nz) break;
            if (cm[d + 1]) {
                phi[c] = v_mask;
                r[c] = 0.0;
                g0[c] = 0.0f;
                continue;
            }
            const double pc = col[d + 1], hr = h2e * rh[d];
            const int nm = mx[d] + mp[d] + my[d] + mq[d] + cm[d] + cm[d + 2];
            const double sum = (i > 0 ? (mx[d] ? v_mask : xm[d]) : pc) + (i < nx - 1 ? (mp[d] ? v_mask : xp[d]) : pc) +
                               (j > 0 ? (my[d] ? v_mask : ym[d]) : pc) + (j < ny - 1 ? (mq[d] ? v_mask : yp[d]) : pc) +
                               (k > 0 ? (cm[d] ? v_mask : col[d]) : 2.0 * v_lo - pc) +
                               (k < nz - 1 ? (cm[d + 2] ? v_mask : col[d + 2]) : 2.0 * v_hi - pc);
            const double rr = hr + sum - 6.0 * pc;
            double b = hr;
            if (k == 0) b += 2.0 * v_lo;
            if (k == nz - 1) b += 2.0 * v_hi;
            if (nm) b += (double)nm * v_mask;
            r[c] = rr;
            g0[c] = (float)rr;
            acc[0] += b * b;
            acc[1] += rr * rr;
        }
    } while (MANY && (k0 += gridDim.z * ZC) < nz);
    double tot[2];
    if (grid_sums64<2>(acc, part, ctr, tot)) {
        sc[S_B2] = tot[0];
        sc[S_R2] = tot[1];
    }
}

// A z of the ZC cells of a thread's column from plane k0 on (0 on electrode
// cells and outside); z is the preconditioned residual (float32, zero on
// electrode cells).  All lanes of a warp (32 consecutive x) call.
struct Apply64 {
    double z[ZC], w[ZC];
};
__device__ __forceinline__ void apply64(const float* __restrict__ z, const uint8_t* __restrict__ mask, int i, int j, int k0,
                                        int nx, int ny, int nz, Apply64& o) {
    const int lane = threadIdx.x, pl = nx * ny;
    const bool in = i < nx && j < ny;
    const int c0 = in ? lin(i, j, 0, nx, ny) : 0;
    float col[ZC + 2], xe[ZC], ym[ZC], yp[ZC];
    uint8_t mk[ZC];
#pragma unroll
    for (int d = 0; d < ZC + 2; ++d) {
        const int k = k0 - 1 + d;
        col[d] = in && k >= 0 && k < nz ? z[c0 + k * pl] : 0.0f;
    }
#pragma unroll
    for (int d = 0; d < ZC; ++d) {
        const int k = k0 + d, c = c0 + k * pl;
        const bool ok = in && k < nz;
        xe[d] = 0.0f;  // the warp's end lanes fetch their outer x neighbour
        if (ok && lane == 0 && i > 0) xe[d] = z[c - 1];
        if (ok && lane == BX - 1 && i < nx - 1) xe[d] = z[c + 1];
        ym[d] = ok && j > 0 ? z[c - nx] : 0.0f;
        yp[d] = ok && j < ny - 1 ? z[c + nx] : 0.0f;
        mk[d] = ok ? mask[c] : 1;
    }
    const double dxy = (double)(6 - ((i == 0) + (i == nx - 1) + (j == 0) + (j == ny - 1)));
    double zd[ZC + 2];
#pragma unroll
    for (int d = 0; d < ZC + 2; ++d) zd[d] = (double)col[d];
#pragma unroll
    for (int d = 0; d < ZC; ++d) {
        const int k = k0 + d;
        double xm = __shfl_up_sync(kFull, zd[d + 1], 1), xp = __shfl_down_sync(kFull, zd[d + 1], 1);
        if (lane == 0) xm = (double)xe[d];
        if (lane == BX - 1) xp = (double)xe[d];
        if (i >= nx - 1) xp = 0.0;
        const double s = ((((xm + xp) + (double)ym[d]) + (double)yp[d]) + zd[d]) + zd[d + 2];
        const double diag = k == 0 || k == nz - 1 ? dxy + 1.0 : dxy;
        o.z[d] = zd[d + 1];
        o.w[d] = mk[d] ? 0.0 : diag * zd[d + 1] - s;
    }
}

// The sums z.r, z.q_prev and z.w with w = A z (stored if w is given), then the
// iteration's scalars (last block).
template <bool MANY>
__global__ void __launch_bounds__(BX * BY) k_apply64(const float* __restrict__ z, const double* __restrict__ r,
                                                     const double* __restrict__ q_prev, double* __restrict__ w,
                                                     const uint8_t* __restrict__ mask, int nx, int ny, int nz, int first,
                                                     double* part, unsigned* ctr, double* sc) {
    pdl_wait();
    const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y;
    const bool in = i < nx && j < ny;
    const int pl = nx * ny, c0 = in ? lin(i, j, 0, nx, ny) : 0;
    double acc[3] = {0.0, 0.0, 0.0};
    int k0 = blockIdx.z * ZC;
    do {
        double rv[ZC], qv[ZC];
#pragma unroll
        for (int d = 0; d < ZC; ++d) {
            const bool ok = in && k0 + d < nz;
            rv[d] = ok ? r[c0 + (k0 + d) * pl] : 0.0;
            qv[d] = ok && !first ? q_prev[c0 + (k0 + d) * pl] : 0.0;
        }
        Apply64 o;
        apply64(z, mask, i, j, k0, nx, ny, nz, o);
#pragma unroll
        for (int d = 0; d < ZC; ++d) {
            if (!in || k0 + d >= nz) break;
            if (w) w[c0 + (k0 + d) * pl] = o.w[d];
            acc[0] += o.z[d] * rv[d];
            if (!first) acc[1] += o.z[d] * qv[d];
            acc[2] += o.z[d] * o.w[d];
        }
    } while (MANY && (k0 += gridDim.z * ZC) < nz);
    double tot[3];
    if (grid_sums64<3>(acc, part, ctr, tot)) cg_scalars(tot, first, sc);
}

// p = z + beta p, q = w + beta q, phi += alpha p, r -= alpha q with its
// float32 copy, ||r||^2.  Without a stored w (MG::carve) w = A z is formed again: the same values, 13 double
// operations a cell more (16 us in place of 7 on 64 x 48 x 80 cells).
template <bool MANY>
__global__ void __launch_bounds__(BX * BY) k_step64(const float* __restrict__ z, const double* __restrict__ w,
                                                    const uint8_t* __restrict__ mask, double* __restrict__ p,
                                                    double* __restrict__ q, double* __restrict__ phi,
                                                    double* __restrict__ r, float* __restrict__ g0, int nx, int ny, int nz,
                                                    int first, double* part, unsigned* ctr, double* sc) {
    pdl_wait();
    const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y;
    const double a = sc[S_ALPHA], b = first ? 0.0 : sc[S_BETA];
    const bool in = i < nx && j < ny, prev = b != 0.0;
    const int pl = nx * ny;
    double acc[1] = {0.0};
    int k0 = blockIdx.z * ZC;
    do {
        const int c0 = in ? lin(i, j, k0, nx, ny) : 0;
        double pv[ZC], qv[ZC], fv[ZC], rv[ZC];
#pragma unroll
        for (int d = 0; d < ZC; ++d) {
            const bool ok = in && k0 + d < nz;
            pv[d] = ok && prev ? p[c0 + d * pl] : 0.0;
            qv[d] = ok && prev ? q[c0 + d * pl] : 0.0;
            fv[d] = ok ? phi[c0 + d * pl] : 0.0;
            rv[d] = ok ? r[c0 + d * pl] : 0.0;
        }
        Apply64 o;
        if (w) {
#pragma unroll
            for (int d = 0; d < ZC; ++d) {
                const bool ok = in && k0 + d < nz;
                o.z[d] = ok ? (double)z[c0 + d * pl] : 0.0;
                o.w[d] = ok ? w[c0 + d * pl] : 0.0;
            }
        } else {
            apply64(z, mask, i, j, k0, nx, ny, nz, o);
        }
#pragma unroll
        for (int d = 0; d < ZC; ++d) {
            if (!in || k0 + d >= nz) break;
            const int c = c0 + d * pl;
            const double pp = prev ? o.z[d] + b * pv[d] : o.z[d], qq = prev ? o.w[d] + b * qv[d] : o.w[d];
            p[c] = pp;
            q[c] = qq;
            phi[c] = fv[d] + a * pp;
            const double rr = rv[d] - a * qq;
            r[c] = rr;
            g0[c] = (float)rr;
            acc[0] += rr * rr;
        }
    } while (MANY && (k0 += gridDim.z * ZC) < nz);
    double tot[1];
    if (grid_sums64<1>(acc, part, ctr, tot)) sc[S_R2] = tot[0];
}

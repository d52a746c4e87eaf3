// The small levels of the multigrid hierarchy in one block (included by
// poisson.cu inside its anonymous namespace).
//
// A thread owns the same cells throughout (of each colour one, on the first
// level up to four): their table words, right-hand sides and reciprocal
// diagonals stay in registers while it works on the level, and e stands in
// shared memory, each colour in an array of its own, so that a warp's cells
// and all their neighbours are consecutive words.  A half-sweep is then six
// shared loads, the arithmetic, a store and a barrier.  Smaller levels use the
// first threads of the block, which meet at named barriers while the others
// wait.  The tables (built with the masks) hold what needs divisions.
//
// What bounds it: the chain of ~45 dependent phases, not the issue rate; a
// phase that looks its cells up again costs 700 to 1800 clocks however few
// cells it has, and code that is unrolled over the levels 1200 (instruction
// fetch).  One launch within a solve, plain kernel and this one: 16^3 .. 2^3
// 23.4 and 12.5 us, 16 x 12 x 20 .. 4 x 3 x 5 24.8 and 10.4, 16 x 16 x 32 .. 2
// x 2 x 4 32.9 and 21.5.  The values are those of the plain kernels, operation
// by operation.
constexpr int kTailMaxLevels = 6;
constexpr int kTailThreads = 1024;
constexpr int kTailPerThread = 4;  // cells of one colour a thread owns at most (first level)
constexpr size_t kTailSmem = 200 * 1024;

// A cell's table entry.
//  x: offset in its colour's e array (bits 0-15), diagonal 2..8 or 0 for a
//     cell held at zero or outside (16-19), parity of its x (20), no neighbour
//     at x - 1 (21) or x + 1 (22), cell exists (23)
//  y: index in the level, x fastest
//  z: index of the coarse cell it lies in (0-15), steps to the near coarse
//     neighbours in x, y, z (16-17, 18-19, 20-21: 0, 1 or 2 for -1), ghost in z (22)
//  w: place of the first red child's residual on the finer level
struct TailLevel {
    int nx, ny, nz, hx;  // hx: slots a row of one colour ((nx + 1) / 2)
    int h;               // slots of one colour (nz ny hx)
    int plane, ca;       // e: pitch of a plane, size of one colour's array (rows and planes of zeros around)
    int e, g, r, p, w;   // shared memory: floats of e, g, residuals, plain copy; entry of the table
    int act;             // threads that work on the level
};
struct TailPlan {
    TailLevel L[kTailMaxLevels];
    float* e_first;        // global e of the first of these levels
    const float* g_first;  // global g of the same
    const uint4* tab;      // tables of all levels
    int levels, words, cells;  // floats of shared memory; table entries
    int pre, post, coarse;
};

__host__ __device__ inline TailLevel tail_geometry(int nx, int ny, int nz) {
    TailLevel L = {};
    L.nx = nx; L.ny = ny; L.nz = nz;
    L.hx = (nx + 1) / 2;
    L.h = nz * ny * L.hx;
    L.plane = (ny + 2) * L.hx;
    L.ca = (nz + 2) * L.plane;
    L.act = L.h < kTailThreads ? (L.h + 31) & ~31 : kTailThreads;
    return L;
}
// Places of the levels: the first level's table and g stay in registers.
__host__ __device__ inline void tail_place(TailPlan& T) {
    int o = 0, c = 0;
    for (int l = 0; l < T.levels; ++l) {
        TailLevel& L = T.L[l];
        L.w = c;
        c += 2 * L.h;
        if (l > 0) o += 8 * L.h;  // table entries, 16 bytes each (at 4 times their index from the first level's end)
    }
    T.cells = c;
    for (int l = 0; l < T.levels; ++l) {
        TailLevel& L = T.L[l];
        L.e = o;
        o += 2 * L.ca;
        L.r = o;
        o += L.h;
        if (l > 0) {
            L.g = o;
            o += 2 * L.h;
            L.p = o;
            o += L.nx * L.ny * L.nz;
        }
    }
    T.words = o;
}

__global__ void k_tail_table(const uint8_t* __restrict__ m, TailLevel L, TailLevel F, uint4* __restrict__ tab) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= 2 * L.h) return;
    const int color = p >= L.h ? 1 : 0, r = p - color * L.h, ii = r % L.hx, j = (r / L.hx) % L.ny, k = r / (L.hx * L.ny);
    const int i = 2 * ii + ((j + k + color) & 1);
    uint4 c = make_uint4((uint32_t)((k + 1) * L.plane + (j + 1) * L.hx + ii), 0u, 0u, 0u);
    if (i < L.nx) {
        const int diag = 6 - ((i == 0) + (i == L.nx - 1) + (j == 0) + (j == L.ny - 1)) + ((k == 0) + (k == L.nz - 1));
        c.y = (uint32_t)((k * L.ny + j) * L.nx + i);
        c.x |= (m[c.y] ? 0u : (uint32_t)diag) << 16;
        c.x |= (uint32_t)(i & 1) << 20 | (i == 0 ? 1u << 21 : 0u) | (i == L.nx - 1 ? 1u << 22 : 0u) | 1u << 23;
        const int cx = L.nx / 2, cy = L.ny / 2, cz = L.nz / 2, I = i >> 1, J = j >> 1, K = k >> 1;
        auto step = [](int odd, int I_, int n) -> uint32_t { return odd ? (I_ + 1 < n ? 1u : 0u) : (I_ > 0 ? 2u : 0u); };
        if (I < cx && J < cy && K < cz) {
            c.z = (uint32_t)((K * cy + J) * cx + I);
            c.z |= step(i & 1, I, cx) << 16 | step(j & 1, J, cy) << 18 | step(k & 1, K, cz) << 20;
            if (step(k & 1, K, cz) == 0u) c.z |= 1u << 22;
        }
        c.w = (uint32_t)((2 * k * F.ny + 2 * j) * F.hx + i);  // F: the finer level (unused on the first)
    }
    tab[p] = c;
}

// A thread's cells of a level, colour by colour.
template <int C> struct TailCells {
    uint32_t w[2][C];
    float g[2][C], r[2][C];
};
__device__ __forceinline__ float tail_rdiag(uint32_t w) {
    const uint32_t d = (w >> 16) & 15u;
    return d ? inv_diag((float)d) : 0.0f;
}

// Neighbour sum of a cell (en: the other colour's e), as nb_sum_e.
__device__ __forceinline__ float tail_sum(int hx, int plane, uint32_t w, const float* en) {
    const int o = w & 0xffffu, b = o + ((w >> 20) & 1u);
    const float xm = (w >> 21) & 1u ? 0.0f : en[b - 1], xp = (w >> 22) & 1u ? 0.0f : en[b];
    return ((((xm + xp) + en[o - hx]) + en[o + hx]) + en[o - plane]) + en[o + plane];
}

template <int C, int COLOR>
__device__ __forceinline__ void tail_half(const TailCells<C>& c, const TailLevel& L, float* e) {
    float* eo = e + COLOR * L.ca;
    const float* en = e + (1 - COLOR) * L.ca;
    float v[C];
#pragma unroll
    for (int u = 0; u < C; ++u) v[u] = (c.g[COLOR][u] + tail_sum(L.hx, L.plane, c.w[COLOR][u], en)) * c.r[COLOR][u];
#pragma unroll
    for (int u = 0; u < C; ++u)
        if ((c.w[COLOR][u] >> 16) & 15u) eo[c.w[COLOR][u] & 0xffffu] = v[u];
}

// n full sweeps red, black; or, from the black side, black, red.
template <int C>
__device__ __forceinline__ void tail_sweeps(const TailCells<C>& c, const TailLevel& L, float* e, int n, bool black_first, int id) {
    const int turns = black_first ? n + 1 : n;
#pragma unroll 1
    for (int s = 0; s < turns; ++s) {
        if (!black_first || s > 0) {
            tail_half<C, 0>(c, L, e);
            bar_named(id, L.act);
        }
        if (!black_first || s < n) {
            tail_half<C, 1>(c, L, e);
            bar_named(id, L.act);
        }
    }
}

// Residuals of the red cells (the black ones are zero after a black half-sweep).
template <int C> __device__ __forceinline__ void tail_resid(const TailCells<C>& c, const TailLevel& L, const float* e, float* R, int t) {
#pragma unroll
    for (int u = 0; u < C; ++u) {
        const uint32_t w = c.w[0][u], d = (w >> 16) & 15u;
        const float s = tail_sum(L.hx, L.plane, w, e + L.ca);
        const float r = c.g[0][u] - ((float)d * e[w & 0xffffu] - s);
        if (t + u * L.act < L.h) R[t + u * L.act] = d ? r : 0.0f;
    }
}

// The red cells take the interpolated correction (weights 3/4, 1/4) from the
// plain copy P of the coarser level's e; the black ones are formed anew by the
// half-sweep that follows, from red neighbours alone.
__device__ __forceinline__ void tail_prolong(uint32_t w, uint32_t z, int cx, int cxy, const float* P, float* e) {
    if (!((w >> 16) & 15u)) return;
    auto sgn = [](uint32_t s) { return s == 2u ? -1 : (int)s; };
    const float* c0 = P + (z & 0xffffu);
    const int dx = sgn((z >> 16) & 3u), dy = sgn((z >> 18) & 3u) * cx, dz = sgn((z >> 20) & 3u) * cxy;
    const float sg = (z >> 22) & 1u ? -1.0f : 1.0f;
    float acc = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int a = u >> 2, b = (u >> 1) & 1, d = u & 1;
        const float wgt = (a ? 0.25f : 0.75f) * (b ? 0.25f : 0.75f) * (d ? 0.25f : 0.75f);
        const float v = c0[(a ? dz : 0) + (b ? dy : 0) + (d ? dx : 0)];
        acc = fmaf(wgt, a ? sg * v : v, acc);
    }
    e[w & 0xffffu] += acc;
}

// C: cells of one colour a thread owns on the first level.
template <int C> __global__ void __launch_bounds__(kTailThreads, 1) k_tail_cycle(const __grid_constant__ TailPlan T) {
    extern __shared__ __align__(16) unsigned char tail_sm[];
    float* sm = reinterpret_cast<float*>(tail_sm);
    uint4* W = reinterpret_cast<uint4*>(tail_sm);  // tables of the levels after the first
    const int t = threadIdx.x, last = T.levels - 1, nthr = blockDim.x;
    const TailLevel L0 = T.L[0];
    // what does not depend on the kernel before: the tables, zeros
    TailCells<C> c;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int u = 0; u < C; ++u) {
            const int p = t + u * nthr;
            // beyond the level: a valid place, held at zero
            c.w[q][u] = p < L0.h ? __ldg(&T.tab[q * L0.h + p].x) : (uint32_t)(L0.plane + L0.hx);
            c.r[q][u] = tail_rdiag(c.w[q][u]);
        }
    const int n1 = T.cells - 2 * L0.h;
    for (int p = t; p < n1; p += nthr) W[p] = __ldg(T.tab + 2 * L0.h + p);
    for (int p = 4 * n1 + t; p < T.words; p += nthr) sm[p] = 0.0f;
    pdl_wait();
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int u = 0; u < C; ++u)
            c.g[q][u] = (c.w[q][u] >> 23) & 1u ? T.g_first[__ldg(&T.tab[q * L0.h + t + u * nthr].y)] : 0.0f;
    __syncthreads();
    float* e0 = sm + L0.e;
    tail_sweeps<C>(c, L0, e0, last == 0 ? T.coarse : T.pre, false, 1);
    if (last > 0) {
        tail_resid<C>(c, L0, e0, sm + L0.r, t);
        bar_named(1, L0.act);
        // the levels below, down and up; a thread goes down to the last one it works on
        int l = 1;
#pragma unroll 1
        for (; l <= last; ++l) {
            const TailLevel L = T.L[l];
            if (t >= L.act) break;
            const TailLevel& F = T.L[l - 1];
            const uint4* Wl = W + (L.w - 2 * L0.h);
            TailCells<1> s;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 cell = t < L.h ? Wl[q * L.h + t] : make_uint4((uint32_t)(L.plane + L.hx), 0u, 0u, 0u);
                const float* R = sm + F.r + cell.w;
                const float acc = (((0.0f + R[0]) + R[F.hx]) + R[F.ny * F.hx]) + R[F.ny * F.hx + F.hx];
                s.w[q][0] = cell.x;
                s.r[q][0] = tail_rdiag(cell.x);
                s.g[q][0] = (cell.x >> 16) & 15u ? 0.5f * acc : 0.0f;
                if (t < L.h) sm[L.g + q * L.h + t] = s.g[q][0];
            }
            float* e = sm + L.e;
            tail_sweeps<1>(s, L, e, l == last ? T.coarse : T.pre, false, l + 1);
            if (l < last) {
                tail_resid<1>(s, L, e, sm + L.r, t);
                bar_named(l + 1, L.act);
            }
        }
#pragma unroll 1
        for (--l; l >= 1; --l) {
            const TailLevel L = T.L[l];
            const uint4* Wl = W + (L.w - 2 * L0.h);
            float* e = sm + L.e;
            if (l < last) {
                bar_named(l + 1, L.act);  // the coarser level is done
                const TailLevel& D = T.L[l + 1];
                TailCells<1> s;
                uint32_t z = 0;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const uint4 cell = t < L.h ? Wl[q * L.h + t] : make_uint4((uint32_t)(L.plane + L.hx), 0u, 0u, 0u);
                    s.w[q][0] = cell.x;
                    s.r[q][0] = tail_rdiag(cell.x);
                    s.g[q][0] = t < L.h ? sm[L.g + q * L.h + t] : 0.0f;
                    if (q == 0) z = cell.z;
                }
                tail_prolong(s.w[0][0], z, D.nx, D.nx * D.ny, sm + D.p, e);
                bar_named(l + 1, L.act);
                tail_sweeps<1>(s, L, e, T.post, true, l + 1);
            }
            // the plain copy for the finer level
            if (t < L.h)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const uint4 cell = Wl[q * L.h + t];
                    if ((cell.x >> 23) & 1u) sm[L.p + cell.y] = e[q * L.ca + (cell.x & 0xffffu)];
                }
        }
        bar_named(1, L0.act);
        const TailLevel& D = T.L[1];
#pragma unroll
        for (int u = 0; u < C; ++u) {
            const int p = t + u * nthr;
            if (p < L0.h) tail_prolong(c.w[0][u], __ldg(&T.tab[p].z), D.nx, D.nx * D.ny, sm + D.p, e0);
        }
        bar_named(1, L0.act);
        tail_sweeps<C>(c, L0, e0, T.post, true, 1);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int u = 0; u < C; ++u)
            if ((c.w[q][u] >> 23) & 1u)
                T.e_first[__ldg(&T.tab[q * L0.h + t + u * nthr].y)] = e0[q * L0.ca + (c.w[q][u] & 0xffffu)];
}

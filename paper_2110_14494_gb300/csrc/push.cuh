// Electron push + null-collision Monte Carlo + fixed-point deposit kernels.
//
// Sec. 2.1.1 of the paper: electrons are advanced with velocity Verlet
// (Eqs. 1-2, a = -(e/m_e) E) and collide with the gas by the null-collision
// method at the constant trial rate nu_max, using rates tabulated from cross
// sections.  Sec. 2.1.3: the field is interpolated to the particle and the
// particle mapped to the grid with trilinear (cloud-in-cell) weights.
//
// A step of an electron: gather, half-kick, the chain of free flights and
// collisions, reflection at the domain faces, electrode absorption, append of
// the survivor to the other buffer with a warp-aggregated cursor, and its
// deposit.  Single precision (collide_loop): one lane owns the electron through
// its flights and collisions.  Double precision (collide_pool): the electron
// stands in its warp's shared memory, and whichever lanes come next do its
// draws and collisions.  Ionization products wait in the warp's queue and fly
// their remaining time as its next work items; k_children finishes those that
// the queue could not take.
// Instantiated for T = float and T = double in separate translation units.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace pic {

enum { MODE_PIC = 0, MODE_SWARM = 1 };
enum { RES_NONE = 0, RES_THIN = 1, RES_DUP = 2 };

template <class T> struct PushArgs {
    Soa<T> in, out;
    ChildQ<T> cq, cq2;         // product queues: parents fill cq; children generation g reads
                               // (g even ? cq : cq2) and spills into the other one
    int gen;
    int sms;                   // multiprocessors of the device (work distribution)
    DevState* st;
    const T* table;            // rate table (see kTableRow)
    int n_bins, n_proc;
    int kind[8];
    T thr[8];                  // eV
    T mratio[8];               // m_e / M (0 = infinite mass)
    T l0, inv_dl;              // ln(eps_0), (n_bins-1) / (ln eps_last - ln eps_0), in T
    T eps_lo, eps_hi;          // eV
    T nu_max;
    T tau_scale;               // flight-time factor (flight_scale)
    T inv_dl2, l0t;            // ln 2 * inv_dl and l0 * inv_dl: table coordinate from a base-2 logarithm
    T dt;                      // duration of this step
    int trip_limit;            // of the collision loops in double precision (trip_limit)
    T dt_kick;                 // duration of the previous step (the half-kick completes its Eq. 2)
    Keys K;
    uint32_t step;
    int first;                 // previous acceleration unknown: no half-kick
    long long cap_out, cap_child;
    // grid (PIC mode)
    int nx, ny, nz;
    T ox, oy, oz, dxr, hx, hy, hz;  // origin, cell size, upper faces
    const T* E4;               // [ncell][4] packed cell-centred field or nullptr (uniform)
    T E0[3];
    const uint8_t* mask;
    unsigned long long *q_e, *q_pos, *q_neg;
    unsigned int* vhist;  // speed histogram of the stored electrons (adaptive time step), or null
    int boundary;
    int axi;                   // axisymmetric grid (see grid_pt)
    // photoionization (Sec. 2.4): emission probability per ionization, the
    // absorption coefficient range [chi_a, chi_a e^chi_log] (1/m), and the
    // queue of photoelectrons appended after the step
    T photo_prob, chi_a, chi_log;
    T *pe_x, *pe_y, *pe_z, *pe_w;   // emitted photons: origin and weight
    uint64_t* pe_id;                // emitting electron and draw index
    uint32_t* pe_k;
    T *ph_x, *ph_y, *ph_z, *ph_w;   // photoelectrons
    uint64_t* ph_id;
    long long cap_photo;
    // swarm mode
    double* mom;               // [kNMom] accumulators of this step
    long long n_lo, n_hi;
};

// Per-process constants, staged in shared memory after the rate table so the
// process index can address them without a local-memory copy of the
// kernel parameters.
template <class T> struct ProcSmem {
    T thr[8];
    T mratio[8];
    int kind[8];
};

// ------------------------------------------------------------------ arithmetic
// Double-precision arithmetic runs on two lanes a clock per multiprocessor,
// so a double operation costs a warp sixteen clocks whatever its lanes do; the
// helpers below give the values of the plain expressions with fewer of them.
// x / c for a constant c with rc = 1 / c rounded to nearest: the quotient's
// estimate is corrected to within one unit in the last place, and the last
// correction by its exact remainder then rounds correctly (Markstein, IBM J.
// Res. Dev. 34, 1990, theorem on division by a correctly rounded reciprocal).
__device__ __forceinline__ double div_const(double x, double c, double rc) {
    double q = __dmul_rn(x, rc);
    q = __fma_rn(__fma_rn(-c, q, x), rc, q);
    return __fma_rn(__fma_rn(-c, q, x), rc, q);
}
// max(x, 0) with dmax's choice for NaN (0): not negative and not NaN as integers.
__device__ __forceinline__ float max0(float x) { return dmax(x, 0.0f); }
__device__ __forceinline__ double max0(double x) {
    return (unsigned long long)__double_as_longlong(x) <= 0x7ff0000000000000ull ? x : 0.0;
}
// a >= b of positive values.
__device__ __forceinline__ bool ge_pos(float a, float b) { return a >= b; }
__device__ __forceinline__ bool ge_pos(double a, double b) { return __double_as_longlong(a) >= __double_as_longlong(b); }

// Double precision follows the oracle's operation order (no FMA contraction in
// that translation unit); single precision uses precomputed factors.
template <class T> struct Arith;
template <> struct Arith<double> {
    static __device__ __forceinline__ double energy(double v2) { return div_const(0.5 * kMe * v2, kQ, 1.0 / kQ); }
    static __device__ __forceinline__ double speed(double e) { return sqrt(div_const(2.0 * kQ * e, kMe, 1.0 / kMe)); }
    static __device__ __forceinline__ double lg(double u) { return log(u); }
    static __device__ __forceinline__ double tau(double u0, double nu_max) { return -log(u0) / nu_max; }
    static __device__ __forceinline__ void sc2pi(double u, double* s, double* c) { sincospi(2.0 * u, s, c); }
};
template <> struct Arith<float> {
    static __device__ __forceinline__ float energy(float v2) { return (float)(0.5 * kMe / kQ) * v2; }
    static __device__ __forceinline__ float speed(float e) { return sqrtf((float)(2.0 * kQ / kMe) * e); }
    static __device__ __forceinline__ float lg(float u) { return logf(u); }
    static __device__ __forceinline__ float tau(float u0, float nu_max) { return -logf(u0) / nu_max; }
    static __device__ __forceinline__ void sc2pi(float u, float* s, float* c) { sincospif(2.0f * u, s, c); }
};

// cos and sin of the polar angle, cos = 1 - 2 u2.  In double precision 2 u2
// and ct^2 are exact (u2 has 24 bits), so each fused operation rounds as the
// two it replaces, and 1 - ct^2 is at least 2^-23.
__device__ __forceinline__ void polar(float u2, float& ct, float& st) {
    ct = 1.0f - 2.0f * u2;
    st = sqrtf(dmax(0.0f, 1.0f - ct * ct));
}
__device__ __forceinline__ void polar(double u2, double& ct, double& st) {
    ct = __fma_rn(-2.0, u2, 1.0);
    st = sqrt(__fma_rn(-ct, ct, 1.0));
}

template <class T> __device__ __forceinline__ void iso_dir(T u2, T u3, T n[3]) {
    T ct, st;
    polar(u2, ct, st);
    T s, c;
    Arith<T>::sc2pi(u3, &s, &c);
    n[0] = st * c;
    n[1] = st * s;
    n[2] = ct;
}

template <class T> __device__ __forceinline__ void fly(T x[3], T v[3], const T a[3], T tau) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // a field along one axis (swarms): the other two only drift
        if (sizeof(T) == 8 && (__double_as_longlong((double)a[d]) << 1) == 0) {
            x[d] = x[d] + tau * v[d];
            continue;
        }
        x[d] = x[d] + tau * (v[d] + (T)0.5 * tau * a[d]);
        v[d] = v[d] + tau * a[d];
    }
}

// ---------------------------------------------------------------- per-thread stats
struct LStats {
    unsigned long long events, nulls, clamped, absorbed, attached, children, processed;
    unsigned long long coll[8];
    double w_ion, w_att, w_abs;
    __device__ void zero() {
        events = nulls = clamped = absorbed = attached = children = processed = 0;
        for (int k = 0; k < 8; ++k) coll[k] = 0;
        w_ion = w_att = w_abs = 0.0;
    }
};

template <class T> struct MomAcc {
    double m[kNMom];
    __device__ void zero() {
        for (int q = 0; q < kNMom; ++q) m[q] = 0.0;
    }
    __device__ void add(const T x[3], const T v[3], T wt) {
        double w = wt, X = x[0], Y = x[1], Z = x[2], U = v[0], V = v[1], W = v[2];
        m[0] += w; m[1] += w * X; m[2] += w * Y; m[3] += w * Z;
        m[4] += w * X * X; m[5] += w * Y * Y; m[6] += w * Z * Z;
        m[7] += w * U; m[8] += w * V; m[9] += w * W;
        m[10] += w * X * U; m[11] += w * Y * V; m[12] += w * Z * W;
        m[13] += w * (0.5 * kMe * (U * U + V * V + W * W) / kQ);
    }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Flushes per-thread statistics (all threads of the block must call).
template <class T>
__device__ void flush_stats(const PushArgs<T>& A, LStats& s, int n_proc) {
    unsigned long long e = warp_sum(s.events), nn = warp_sum(s.nulls), cl = warp_sum(s.clamped);
    unsigned long long ab = warp_sum(s.absorbed), at = warp_sum(s.attached), ch = warp_sum(s.children);
    unsigned long long pr = warp_sum(s.processed);
    double wi = warp_sum(s.w_ion), wa = warp_sum(s.w_att), wb = warp_sum(s.w_abs);
    unsigned long long co[8];
    for (int k = 0; k < 8; ++k) co[k] = warp_sum(s.coll[k]);
    if ((threadIdx.x & 31) == 0) {
        DevState* st = A.st;
        if (e) atomicAdd(&st->n_events, e);
        if (nn) atomicAdd(&st->n_null, nn);
        if (cl) atomicAdd(&st->n_clamped, cl);
        if (ab) atomicAdd(&st->n_absorbed, ab);
        if (at) atomicAdd(&st->n_attached, at);
        if (ch) atomicAdd(&st->n_children, ch);
        if (pr) atomicAdd(&st->n_processed, pr);
        for (int k = 0; k < n_proc && k < 8; ++k)
            if (co[k]) atomicAdd(&st->n_coll[k], co[k]);
        if (wi != 0.0) atomicAdd(&st->w_ion, wi);
        if (wa != 0.0) atomicAdd(&st->w_att, wa);
        if (wb != 0.0) atomicAdd(&st->w_absorbed, wb);
    }
}

template <class T>
__device__ void flush_moments(const PushArgs<T>& A, MomAcc<T>& M, double* red /* smem [kNMom][32] */) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int q = 0; q < kNMom; ++q) {
        double v = warp_sum(M.m[q]);
        if (lane == 0) red[q * 32 + wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < kNMom) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) s += red[threadIdx.x * 32 + w];
        if (s != 0.0) atomicAdd(&A.mom[threadIdx.x], s);
    }
}

// ------------------------------------------------------------------ gather
template <class T>
__device__ __forceinline__ void axis_w(T x, T o, T dx, int n, int& i0, int& i1, T& f) {
    T s = (x - o) / dx - (T)0.5;
    if (s < (T)0) s = (T)0;
    if (s > (T)(n - 1)) s = (T)(n - 1);
    int i = (int)floor(s);
    if (i > n - 2) i = n - 2;
    if (i < 0) i = 0;
    i0 = i;
    i1 = i + 1;
    f = s - (T)i;
}

template <class T> struct Ld4;
template <> struct Ld4<float> {
    static __device__ __forceinline__ void get(const float* p, float e[3]) {
        float4 v = __ldg(reinterpret_cast<const float4*>(p));
        e[0] = v.x; e[1] = v.y; e[2] = v.z;
    }
};
template <> struct Ld4<double> {
    static __device__ __forceinline__ void get(const double* p, double e[3]) {
        double2 a = __ldg(reinterpret_cast<const double2*>(p));
        double b = __ldg(p + 2);
        e[0] = a.x; e[1] = a.y; e[2] = b;
    }
};

// Point of the grid that a particle position maps to.  Cartesian grids: the
// position itself.  Axisymmetric grids (Sec. 2.1.1: particles move in 3D,
// the field and densities live on an (r, z) mesh): (r, centre of the single
// y cell, z) with r = sqrt(x^2 + y^2), so cell indices, deposits and masks of
// the Cartesian code address the ring cell (i_r, 0, k).
template <class T> __device__ __forceinline__ void grid_pt(const PushArgs<T>& A, const T x[3], T g[3]) {
    if (A.axi) {
        g[0] = sqrt(x[0] * x[0] + x[1] * x[1]);
        g[1] = A.oy + (T)0.5 * A.dxr;
        g[2] = x[2];
    } else {
        g[0] = x[0]; g[1] = x[1]; g[2] = x[2];
    }
}

// Axisymmetric gather: E_r and E_z bilinear in (r, z) at cell centres
// (packed as (E_r, 0, E_z)), projected on x and y: E = (E_r x / r, E_r y / r,
// E_z) (Sec. 2.1.1), zero radial part on the axis.
template <class T>
__device__ __forceinline__ void gather_axi(const PushArgs<T>& A, const T x[3], T E[3]) {
    const T r = sqrt(x[0] * x[0] + x[1] * x[1]);
    int ir[2], iz[2];
    T fr, fz;
    axis_w(r, A.ox, A.dxr, A.nx, ir[0], ir[1], fr);
    axis_w(x[2], A.oz, A.dxr, A.nz, iz[0], iz[1], fz);
    const T gr[2] = {(T)1 - fr, fr}, gz[2] = {(T)1 - fz, fz};
    T er = (T)0, ez = (T)0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int dz = c >> 1, dr = c & 1;
        const long long idx = (long long)iz[dz] * A.nx + ir[dr];
        T e[3];
        Ld4<T>::get(A.E4 + 4 * idx, e);
        const T g = gz[dz] * gr[dr];
        er += g * e[0];
        ez += g * e[2];
    }
    const T inv = r > (T)0 ? er / r : (T)0;
    E[0] = inv * x[0];
    E[1] = inv * x[1];
    E[2] = ez;
}

template <class T>
__device__ __forceinline__ void gather(const PushArgs<T>& A, const T x[3], T E[3]) {
    if (A.E4 == nullptr) { E[0] = A.E0[0]; E[1] = A.E0[1]; E[2] = A.E0[2]; return; }
    if (A.axi) { gather_axi(A, x, E); return; }
    int ix[2], iy[2], iz[2];
    T fx, fy, fz;
    axis_w(x[0], A.ox, A.dxr, A.nx, ix[0], ix[1], fx);
    axis_w(x[1], A.oy, A.dxr, A.ny, iy[0], iy[1], fy);
    axis_w(x[2], A.oz, A.dxr, A.nz, iz[0], iz[1], fz);
    const T gx[2] = {(T)1 - fx, fx}, gy[2] = {(T)1 - fy, fy}, gz[2] = {(T)1 - fz, fz};
    T acc[3] = {(T)0, (T)0, (T)0};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int dz = c >> 2, dy = (c >> 1) & 1, dxx = c & 1;
        const long long idx = ((long long)iz[dz] * A.ny + iy[dy]) * A.nx + ix[dxx];
        T e[3];
        Ld4<T>::get(A.E4 + 4 * idx, e);
        const T g = (gz[dz] * gy[dy]) * gx[dxx];
#pragma unroll
        for (int d = 0; d < 3; ++d) acc[d] += g * e[d];
    }
    E[0] = acc[0]; E[1] = acc[1]; E[2] = acc[2];
}

// ------------------------------------------------------------------ deposit
// Fixed-point cloud-in-cell: S = 2^32 per unit weight; corners 0..6 rounded to
// nearest even, corner 7 the remainder, so each particle adds exactly
// rint(w S).  Products are separately rounded (explicit _rn intrinsics).
__device__ __forceinline__ long long rint_ll(float v) { return __float2ll_rn(v); }
__device__ __forceinline__ long long rint_ll(double v) { return __double2ll_rn(v); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float div_rn(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ double div_rn(double a, double b) { return __ddiv_rn(a, b); }

template <class T>
__device__ __forceinline__ void deposit(const T x, const T y, const T z, const T w, T ox, T oy, T oz, T dx, int nx,
                                        int ny, int nz, unsigned long long* q, DevState* st) {
    const T sx = sub_rn(div_rn(sub_rn(x, ox), dx), (T)0.5);
    const T sy = sub_rn(div_rn(sub_rn(y, oy), dx), (T)0.5);
    const T sz = sub_rn(div_rn(sub_rn(z, oz), dx), (T)0.5);
    const T flx = floor(sx), fly = floor(sy), flz = floor(sz);
    const T fx = sub_rn(sx, flx), fy = sub_rn(sy, fly), fz = sub_rn(sz, flz);
    const int i0 = (int)flx, j0 = (int)fly, k0 = (int)flz;
    const T gx[2] = {sub_rn((T)1, fx), fx}, gy[2] = {sub_rn((T)1, fy), fy}, gz[2] = {sub_rn((T)1, fz), fz};
    const T wS = mul_rn(w, (T)4294967296.0);
    if (!(wS < (T)4.0e18)) { atomicOr(&st->err, kErrOverflow); return; }
    long long sum = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int dz = c >> 2, dy = (c >> 1) & 1, dxx = c & 1;
        long long qc;
        if (c < 7) {
            qc = rint_ll(mul_rn(mul_rn(mul_rn(wS, gz[dz]), gy[dy]), gx[dxx]));
            sum += qc;
        } else {
            qc = rint_ll(wS) - sum;
        }
        const int ii = fold_idx(i0 + dxx, nx), jj = fold_idx(j0 + dy, ny), kk = fold_idx(k0 + dz, nz);
        if (qc != 0) atomicAdd(q + (((long long)kk * ny + jj) * nx + ii), (unsigned long long)qc);
    }
}

// Deposit of weight w at particle position x (through grid_pt).
template <class T>
__device__ __forceinline__ void deposit_at(const PushArgs<T>& A, T x0, T x1, T x2, T w, unsigned long long* q) {
    const T x[3] = {x0, x1, x2};
    T g[3];
    grid_pt(A, x, g);
    deposit(g[0], g[1], g[2], w, A.ox, A.oy, A.oz, A.dxr, A.nx, A.ny, A.nz, q, A.st);
}

// ------------------------------------------------------------------ rates
// Arithmetic of one candidate collision.  Double precision follows the
// oracle's operations.  Single precision takes the hardware base-2 logarithm
// (absolute error near 1e-7) and multiplies by precomputed constants instead
// of dividing: a flight time then carries an absolute error near 1e-7 / nu_max
// (far below a cell crossing), a table coordinate one near 1e-5 of a bin, and
// the scattering cosine a reciprocal square root.
// The collision rates a candidate event is tested against: the table
// (see kTableRow), its maximum total nu_max and the flight_scale of that.  One gas for a PIC context; batched swarms of different
// compositions each have their own.
// Factor of the flight times: -ln 2 / nu_max in single precision (times a
// base-2 logarithm), 1 / nu_max in double (div_const).
template <class T> inline T flight_scale(double nu_max) {
    return (T)((sizeof(T) == 4 ? -0.69314718055994530942 : 1.0) / nu_max);
}
template <class T> struct Rates {
    const T* tab;
    T nu_max, tau_scale;
};

template <class T> struct EvArith;
template <> struct EvArith<double> {
    static __device__ __forceinline__ double flight(const Rates<double>& R, double u0) {
        return div_const(-log(u0), R.nu_max, R.tau_scale);
    }
    static __device__ __forceinline__ double coord(const PushArgs<double>& A, double e) {
        return (log(e) - A.l0) * A.inv_dl;
    }
    static __device__ __forceinline__ double cosine(double dot, double v2) {
        const double sp = sqrt(v2);
        return sp > 0.0 ? dot / sp : 0.0;
    }
};
template <> struct EvArith<float> {
    static __device__ __forceinline__ float flight(const Rates<float>& R, float u0) {
        return __fmul_rn(__log2f(u0), R.tau_scale);
    }
    static __device__ __forceinline__ float coord(const PushArgs<float>& A, float e) {
        return fmaf(__log2f(e), A.inv_dl2, -A.l0t);
    }
    static __device__ __forceinline__ float cosine(float dot, float v2) { return v2 > 0.0f ? dot * rsqrtf(v2) : 0.0f; }
};

// Coordinate in the table, linear in ln(eps), clamped at both ends.
template <class T> __device__ __forceinline__ T table_pos(const PushArgs<T>& A, T e, LStats& ls) {
    if (e <= A.eps_lo) {
        if (e < A.eps_lo) ++ls.clamped;
        return (T)0;
    }
    if (e >= A.eps_hi) {
        if (e > A.eps_hi) ++ls.clamped;
        return (T)(A.n_bins - 1);
    }
    return EvArith<T>::coord(A, e);
}
// Its node and the fraction towards the next one.
template <class T> __device__ __forceinline__ void table_split(const PushArgs<T>& A, T t, int& j, T& f) {
    if (sizeof(T) == 8) {
        // floor by adding 1.5 2^52 rounded down: the integer stands in the low word
        const double big = 6755399441055744.0, r = __dadd_rd((double)t, big);
        const int j0 = __double2loint(r);
        j = j0 > A.n_bins - 2 ? A.n_bins - 2 : (j0 < 0 ? 0 : j0);
        f = t - (j == j0 ? (T)(r - big) : (T)j);
        return;
    }
    int jj = (int)floor(t);
    if (jj > A.n_bins - 2) jj = A.n_bins - 2;
    if (jj < 0) jj = 0;
    j = jj;
    f = t - (T)jj;
}

// Two consecutive rows of a table, and one pair of its totals.
template <class T> struct LdTab;
template <> struct LdTab<float> {
    static __device__ __forceinline__ void rows(const float* p, float a[8], float b[8]) {
        const float4* q = reinterpret_cast<const float4*>(p);
        const float4 v0 = __ldg(q), v1 = __ldg(q + 1), v2 = __ldg(q + 2), v3 = __ldg(q + 3);
        a[0] = v0.x; a[1] = v0.y; a[2] = v0.z; a[3] = v0.w; a[4] = v1.x; a[5] = v1.y; a[6] = v1.z; a[7] = v1.w;
        b[0] = v2.x; b[1] = v2.y; b[2] = v2.z; b[3] = v2.w; b[4] = v3.x; b[5] = v3.y; b[6] = v3.z; b[7] = v3.w;
    }
    static __device__ __forceinline__ void pair(const float* p, float& a, float& d) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        a = v.x; d = v.y;
    }
};
template <> struct LdTab<double> {
    static __device__ __forceinline__ void rows(const double* p, double a[8], double b[8]) {
        const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double2 u = __ldg(q + i), v = __ldg(q + 4 + i);
            a[2 * i] = u.x; a[2 * i + 1] = u.y;
            b[2 * i] = v.x; b[2 * i + 1] = v.y;
        }
    }
    static __device__ __forceinline__ void pair(const double* p, double& a, double& d) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(p));
        a = v.x; d = v.y;
    }
};

// A candidate collision that may be real: the table coordinate of the energy
// before it, the rate u1 nu_max to compare with, and the words of the
// scattering direction (few values: they are held through the draws of the
// warp's other lanes).
template <class T> struct Hit {
    T t, target;
    uint32_t z, w;
};

// Chooses the process of a candidate collision: the smallest k with
// u1 nu_max < sum_{i<=k} nu_i(eps); -1 = null collision.  Every process is
// visited by every lane (the same sums in the same order; rows of fewer than
// seven processes end in zeros, which change no sum), so the lanes of a warp
// stay together whichever process they pick.
template <class T> __device__ __forceinline__ int select_process(const PushArgs<T>& A, const Rates<T>& R, const Hit<T>& h) {
    int j;
    T f, a[kTableRow], b[kTableRow];
    table_split(A, h.t, j, f);
    LdTab<T>::rows(R.tab + j * kTableRow, a, b);
    T cum = (T)0;
    int sel = -1;
#pragma unroll
    for (int k = 0; k < kTableRow - 1; ++k) {
        cum += a[k] + f * (b[k] - a[k]);
        sel = (sel < 0 && h.target < cum) ? k : sel;
    }
    return sel;
}

// ------------------------------------------------------------------ flight
// The product of an ionization by draw k of electron `pid`: id from the
// derived-id stream, isotropic direction from its own draw k = 0, speed sp.
template <class T>
__device__ __forceinline__ uint64_t make_child(const Keys& K, uint32_t step, uint64_t pid, uint32_t k, T sp, T vc[3]) {
    const uint64_t cid = derived_id(K, pid, step, 0x80000000u | k);
    const u32x4 rb = draw_words(K, cid, step, 0u);
    T nb[3];
    iso_dir(unif<T>(rb.z), unif<T>(rb.w), nb);
    vc[0] = sp * nb[0]; vc[1] = sp * nb[1]; vc[2] = sp * nb[2];
    return cid;
}

// One electron in flight on a lane: start position x, displacement d within
// the step (x + d is the position; single precision keeps the resolution of
// the short flights that way), velocity, acceleration, weight, remaining time
// and the index k of its next draw.
template <class T> struct Lane {
    T x[3], d[3], v[3], a[3];
    T w, t_left;
    uint64_t id;
    uint32_t k;
};

enum { EV_CONTINUE = 0, EV_DONE = 1, EV_ATTACHED = 2, EV_IONIZED = 3, EV_HIT = 4 };

// Electrode mask of the cell containing x (cell index by correctly rounded
// (x - origin) / dx, folded into the grid).
template <class T> __device__ __forceinline__ bool masked_at(const PushArgs<T>& A, const T xp[3]) {
    T x[3];
    grid_pt(A, xp, x);
    const int i = fold_idx((int)floor(div_rn(sub_rn(x[0], A.ox), A.dxr)), A.nx);
    const int j = fold_idx((int)floor(div_rn(sub_rn(x[1], A.oy), A.dxr)), A.ny);
    const int k = fold_idx((int)floor(div_rn(sub_rn(x[2], A.oz), A.dxr)), A.nz);
    return A.mask[((long long)k * A.ny + j) * A.nx + i] != 0;
}

// Photon of an ionization event (Sec. 2.4, discrete Monte Carlo model), in
// two parts.  In the collision loop only the emission test: draw (id, step,
// 0xD0000000 | k) of the event's draw index k, u0 < photo_prob emits one
// photon of the electron's weight; an emitted photon's origin (position,
// weight, id, k) goes to a queue.  After each launch k_photo_resolve draws
// its path: the absorption coefficient chi log-uniform on [a, b] (u1) and an
// exponential path with rate chi (u2).  This mixture has exactly Zheleznyak's
// absorption density: f(r) = (e^-ar - e^-br) / (r ln(b/a)) = integral over
// chi in [a, b] of [1 / (chi ln(b/a))] chi e^(-chi r).  Direction: cos(theta)
// = 1 - 2 u3 and azimuth 2 pi u0' of draw (id, step, 0xE0000000 | k).  A
// photon absorbed inside the domain and outside the electrode records a
// positive ion there and queues a photoelectron (id derived with tag
// 0xD0000000 | k).
template <class T>
__device__ __forceinline__ void photo_test(const PushArgs<T>& A, const Keys& K, uint32_t step, uint64_t id,
                                           uint32_t k, const T x[3], T w) {
    const u32x4 r = draw_words(K, id, step, 0xD0000000u | k);
    if (!(unif<T>(r.x) < A.photo_prob)) return;
    const unsigned long long slot = atomicAdd(&A.st->n_photo_src, 1ull);
    if ((long long)slot >= A.cap_photo) {
        atomicOr(&A.st->err, kErrPhotoCapacity);
        return;
    }
    A.pe_x[slot] = x[0];
    A.pe_y[slot] = x[1];
    A.pe_z[slot] = x[2];
    A.pe_w[slot] = w;
    A.pe_id[slot] = id;
    A.pe_k[slot] = k;
}

// One draw of the null-collision method (Sec. 2.1.1): flight time tau =
// -ln(u0) / nu_max; if it ends the step, fly to the end (EV_DONE); else fly
// tau and compare u1 nu_max with the total rate at the electron's energy:
// EV_CONTINUE for a null collision, EV_HIT when a process may take it (h;
// without FAST always: select_process then decides).
template <class T, bool FAST>
__device__ __forceinline__ int candidate(const PushArgs<T>& A, const Rates<T>& R, const Keys& K, uint32_t step,
                                         Lane<T>& L, LStats& ls, Hit<T>& h) {
    const u32x4 r = draw_words(K, L.id, step, L.k);
    ++L.k;
    const T tau = EvArith<T>::flight(R, unif<T>(r.x));
    if (ge_pos(tau, L.t_left)) { fly(L.d, L.v, L.a, L.t_left); return EV_DONE; }
    fly(L.d, L.v, L.a, tau);
    L.t_left = sub_rn(L.t_left, tau);
    ++ls.events;
    const T* v = L.v;
    const T v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    h.t = table_pos(A, Arith<T>::energy(v2), ls);
    h.target = unif<T>(r.y) * R.nu_max;
    h.z = r.z;
    h.w = r.w;
    if (FAST) {
        // single precision: the interpolated total decides null collisions
        int j;
        T f, t0, dt;
        table_split(A, h.t, j, f);
        LdTab<T>::pair(R.tab + A.n_bins * kTableRow + 2 * j, t0, dt);
        if (h.target >= t0 + f * dt) { ++ls.nulls; return EV_CONTINUE; }
    }
    return EV_HIT;
}

// The collision of a hit: the process, then isotropic scattering with u2, u3.
// Ionization returns EV_IONIZED with the product's speed in sp (the caller
// queues the product, which flies the remaining time, and its positive-ion
// event); attachment returns EV_ATTACHED (the caller records the negative-ion
// event at the electron's position) and ends the electron.
template <class T, int MODE, bool STATS>
__device__ __forceinline__ int collide(const PushArgs<T>& A, const Rates<T>& R, const ProcSmem<T>* ps, const Hit<T>& h,
                                       Lane<T>& L, LStats& ls, T& sp) {
    const int p = select_process<T>(A, R, h);
    if (p < 0) { ++ls.nulls; return EV_CONTINUE; }
    if (STATS) ++ls.coll[p & 7];
    const int kind = ps->kind[p];
    if (kind == PIC_PROC_ATTACHMENT) {
        if (MODE == MODE_SWARM || STATS) ls.w_att += (double)L.w;
        ++ls.attached;
        return EV_ATTACHED;
    }
    T* v = L.v;
    const T v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2], e = Arith<T>::energy(v2);
    T n[3];
    iso_dir(unif<T>(h.z), unif<T>(h.w), n);
    // energy after the collision: elastic recoil with cos(chi) = n_old . n_new,
    // excitation loss, or half of what ionization leaves (all three formed,
    // one kept: no branch on the process kind)
    const T cchi = EvArith<T>::cosine(v[0] * n[0] + v[1] * n[1] + v[2] * n[2], v2);
    const T e_el = max0(e * ((T)1 - (T)2 * ps->mratio[p] * ((T)1 - cchi)));
    const T e_in = max0(e - ps->thr[p]);
    const T e2 = kind == PIC_PROC_ELASTIC ? e_el : (kind == PIC_PROC_EXCITATION ? e_in : (T)0.5 * e_in);
    const T sp2 = Arith<T>::speed(e2);
    v[0] = sp2 * n[0]; v[1] = sp2 * n[1]; v[2] = sp2 * n[2];
    if (kind == PIC_PROC_IONIZATION) {
        sp = sp2;
        if (MODE == MODE_SWARM || STATS) ls.w_ion += (double)L.w;
        return EV_IONIZED;
    }
    return EV_CONTINUE;
}

// The next draws of a warp's electrons (all lanes call; `active` ones have an
// electron).  Single precision: two draws, the second by the lanes whose first
// was a null collision, then the collisions of all hits together: six of ten
// draws are null, and a warp pays for a collision whatever its lanes.  Double
// precision (batched swarms; a single population: collide_pool): two rounds of
// a draw and its collision (both cost the same on the narrow double pipe, so a
// draw with fewer lanes gains nothing).  Measured per
// pass, 1e6 electrons, float: two draws 330 us, three 355, two rounds 390;
// 1.4e4 electrons, double: two rounds 579 us a step, two draws 610.
template <class T, int MODE, bool FAST, bool STATS>
__device__ __forceinline__ int advance(const PushArgs<T>& A, const Rates<T>& R, const Keys& K, uint32_t step,
                                       const ProcSmem<T>* ps, bool active, Lane<T>& L, LStats& ls, T& sp) {
    constexpr int kRounds = FAST ? 1 : 2, kDraws = FAST ? 2 : 1;
    int r = EV_CONTINUE;
#pragma unroll
    for (int q = 0; q < kRounds; ++q) {
        Hit<T> h;
#pragma unroll
        for (int d = 0; d < kDraws; ++d) {
            if (active && r == EV_CONTINUE) r = candidate<T, FAST>(A, R, K, step, L, ls, h);
            __syncwarp();
        }
        if (r == EV_HIT) r = collide<T, MODE, STATS>(A, R, ps, h, L, ls, sp);
        __syncwarp();
    }
    return r;
}

// Domain faces (specular reflection or absorption) and electrode cells.
template <class T>
__device__ __forceinline__ bool boundaries(const PushArgs<T>& A, T x[3], T v[3], T w, LStats& ls) {
    const T lo[3] = {A.ox, A.oy, A.oz}, hi[3] = {A.hx, A.hy, A.hz};
    bool out = false;
    if (A.axi) {
        // the cylinder r = R of an axisymmetric grid: outflow, or specular
        // reflection (r -> 2R - r, radial velocity reversed)
        const T R = A.hx;
        T r = sqrt(x[0] * x[0] + x[1] * x[1]);
        if (A.boundary == 1) {
            if (r > R) out = true;
        } else {
            for (int it = 0; it < 8 && r > R; ++it) {
                const T rn = (T)2 * R - r, s = rn / r;
                const T ux = x[0] / r, uy = x[1] / r;
                const T vr = v[0] * ux + v[1] * uy;
                x[0] *= s;
                x[1] *= s;
                v[0] -= (T)2 * vr * ux;
                v[1] -= (T)2 * vr * uy;
                r = fabs(rn);
            }
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (A.axi && d < 2) continue;
        if (A.boundary == 1) {
            if (x[d] < lo[d] || x[d] > hi[d]) out = true;
            continue;
        }
        for (int it = 0; it < 8 && (x[d] < lo[d] || x[d] > hi[d]); ++it) {
            if (x[d] < lo[d]) x[d] = (T)2 * lo[d] - x[d];
            else x[d] = (T)2 * hi[d] - x[d];
            v[d] = -v[d];
        }
        if (x[d] < lo[d]) x[d] = lo[d];
        if (x[d] > hi[d]) x[d] = hi[d];
    }
    if (!out && A.mask && masked_at(A, x)) out = true;
    if (out) { ++ls.absorbed; ls.w_abs += (double)w; }
    return !out;
}

template <class T>
__device__ __forceinline__ void store(const Soa<T>& o, unsigned long long s, const T x[3], const T v[3], const T a[3],
                                      T w, uint64_t id) {
    o.r[PX][s] = x[0]; o.r[PY][s] = x[1]; o.r[PZ][s] = x[2];
    o.r[VX][s] = v[0]; o.r[VY][s] = v[1]; o.r[VZ][s] = v[2];
    o.r[AX][s] = a[0]; o.r[AY][s] = a[1]; o.r[AZ][s] = a[2];
    o.r[PW][s] = w; o.id[s] = id;
}

// A swarm's acceleration: the uniform field, no half-kick (a pass of its own
// over the electrons, and the launch that took the resampled count over, cost
// a step of 1e4 electrons 7 of 230 us in double precision, 4 of 75 in single).
template <class T> __device__ __forceinline__ void uniform_accel(const PushArgs<T>& A, T* f) {
    const T qm = (T)(kQ / kMe);
#pragma unroll
    for (int d = 0; d < 3; ++d) f[AX + d] = -qm * A.E0[d];
}

// Work items of a launch's parents: a swarm that k_resample has doubled counts twice its electrons (k_end_step
// takes the count over).
template <int MODE> __device__ __forceinline__ unsigned long long parent_items(const DevState* st) {
    return MODE == MODE_SWARM && st->n_extra ? st->n_extra : st->n_in;
}

// Sec. 2.1.1, Eq. 2: a_new = -(e/m_e) E(x) from the trilinear gather; the
// half-kick v += dt/2 (a_new - a_old) completes the previous step's velocity
// update (skipped when a_old is unknown); a_old <- a_new.  For one loaded
// electron (f = x y z vx vy vz ax ay az w), done by the collision kernel as it
// stages its parents.
template <class T> __device__ __forceinline__ void half_kick(const PushArgs<T>& A, T f[10]) {
    const T qm = (T)(kQ / kMe);
    T E[3];
    gather(A, f, E);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const T an = -qm * E[d];
        if (!A.first) f[VX + d] = f[VX + d] + (T)0.5 * A.dt_kick * (an - f[AX + d]);
        f[AX + d] = an;
    }
}

// Path of every photon emitted in the launch before (see photo_test): the
// absorbed ones inside the gas deposit their ion and queue a photoelectron.
template <class T>
__global__ void __launch_bounds__(256) k_photo_resolve(const PushArgs<T> A) {
    const unsigned long long nq = A.st->n_photo_src;
    const long long n = (long long)nq < A.cap_photo ? (long long)nq : A.cap_photo;
    const uint32_t step = A.step;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const uint64_t id = A.pe_id[i];
        const uint32_t k = A.pe_k[i];
        const T w = A.pe_w[i];
        const u32x4 r = draw_words(A.K, id, step, 0xD0000000u | k);
        const T chi = A.chi_a * exp(unif<T>(r.y) * A.chi_log);
        const T dist = -log(unif<T>(r.z)) / chi;
        const u32x4 r2 = draw_words(A.K, id, step, 0xE0000000u | k);
        T n3[3];
        iso_dir(unif<T>(r.w), unif<T>(r2.x), n3);
        const T xp[3] = {A.pe_x[i] + dist * n3[0], A.pe_y[i] + dist * n3[1], A.pe_z[i] + dist * n3[2]};
            const T lo[3] = {A.ox, A.oy, A.oz}, hi[3] = {A.hx, A.hy, A.hz};
        bool in = true;
        for (int d = A.axi ? 2 : 0; d < 3; ++d)
            if (!(xp[d] >= lo[d] && xp[d] <= hi[d])) in = false;
        if (A.axi && !(sqrt(xp[0] * xp[0] + xp[1] * xp[1]) <= A.hx)) in = false;
        if (!in || (A.mask && masked_at(A, xp))) continue;
        if (A.q_pos) deposit_at(A, xp[0], xp[1], xp[2], w, A.q_pos);
        const unsigned long long slot = atomicAdd(&A.st->n_photo, 1ull);
        if ((long long)slot >= A.cap_photo) {
            atomicOr(&A.st->err, kErrPhotoCapacity);
            continue;
        }
        A.ph_x[slot] = xp[0];
        A.ph_y[slot] = xp[1];
        A.ph_z[slot] = xp[2];
        A.ph_w[slot] = w;
        A.ph_id[slot] = derived_id(A.K, id, step, 0xD0000000u | k);
    }
}

// Photoelectrons queued by k_photo_resolve join the output buffer at rest, with
// the acceleration of the field at their position (so the next step's
// half-kick adds nothing they did not experience), and their charge is
// deposited with the electrons of the step.
template <class T>
__global__ void __launch_bounds__(256) k_photo_append(const PushArgs<T> A) {
    const unsigned long long nq = A.st->n_photo;
    const long long n = (long long)nq < A.cap_photo ? (long long)nq : A.cap_photo;
    const T qm = (T)(kQ / kMe);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const T x[3] = {A.ph_x[i], A.ph_y[i], A.ph_z[i]};
        const T w = A.ph_w[i];
        T E[3];
        gather(A, x, E);
        const T v[3] = {(T)0, (T)0, (T)0};
        const T a[3] = {-qm * E[0], -qm * E[1], -qm * E[2]};
        const unsigned long long slot = atomicAdd(&A.st->n_out, 1ull);
        if ((long long)slot >= A.cap_out) {
            atomicOr(&A.st->err, kErrOutCapacity);
            continue;
        }
        store(A.out, slot, x, v, a, w, A.ph_id[i]);
        if (A.q_e) deposit_at(A, x[0], x[1], x[2], w, A.q_e);
        if (A.vhist && w > (T)0) atomicAdd(&A.vhist[0], 1u);  // at rest: the lowest speed bin
    }
}

// Closes the photoelectron queue of the launch before.
static __global__ void k_photo_done(DevState* st, long long cap) {
    const unsigned long long n = st->n_photo;
    st->n_photons += n < (unsigned long long)cap ? n : (unsigned long long)cap;
    st->n_photo = 0;
    st->n_photo_src = 0;
}

// Swarm resampling in place (decided from the count after the previous step):
// above n_hi each electron survives with probability 1/2 (draw keyed by id,
// step and 0xA0000000), the others get weight 0; below n_lo every electron
// gets a copy with a derived id, appended after the last one.  Weights are
// not rescaled: the coefficients are ratios of moments of the same step.
template <class T>
__global__ void k_resample(const PushArgs<T> A) {
    const long long n = (long long)A.st->n_in;
    const bool thin = n > A.n_hi, dup = n > 0 && n < A.n_lo;
    if (!thin && !dup) return;
    if (dup && 2 * n > A.cap_out) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&A.st->err, kErrOutCapacity);
        return;
    }
    const Soa<T>& p = A.in;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (thin) {
            const u32x4 r = draw_words(A.K, p.id[i], A.step, 0xA0000000u);
            if (!(unif<T>(r.x) < (T)0.5)) p.r[PW][i] = (T)0;
        } else {
            const long long j = n + i;
            for (int f = 0; f < 10; ++f) p.r[f][j] = p.r[f][i];
            p.id[j] = derived_id(A.K, p.id[i], A.step, 0xA0000000u);
        }
    }
    if (dup && blockIdx.x == 0 && threadIdx.x == 0) A.st->n_extra = (unsigned long long)(2 * n);
}

// ------------------------------------------------------------------ collisions
// Single precision (collide_loop; double precision: collide_pool, which has the
// output stage and the product queue in common): lanes refill from per-warp
// shared-memory stages.  Every lane owns one electron at a time and advances it by up to two draws and a
// collision per loop iteration (advance); a lane whose electron has finished
// the step takes the next electron from the warp's input stage at once, so the
// warp stays converged while electrons need different numbers of events.  All
// per-electron memory work is done by the whole warp, 32 electrons at a time:
// the input stage is filled with one coalesced load of consecutive work items,
// finished electrons wait in the output stage until 32 are there and are then
// reflected at the faces, tested against the electrode, appended with one
// cursor increment, stored and deposited by 32 lanes together.  An ionization
// product waits as a compact entry in the warp's queue and is built (derived
// id, direction from its own draw, positive-ion event of its birth) with 31
// others as the stage's next work items; it flies the remaining time with the
// acceleration of the electron that ionized.  A product that finds the queue
// full waits in the queue of the next (children) launch.
//
// CHILD = false: work item = one electron of the input buffer, kicked as it is
// staged and flying dt.  CHILD = true: work item = one queued ionization
// product, built when it is staged.
constexpr int kRow = 11;    // padded row of a stage entry: x y z vx vy vz ax ay az w t
constexpr int kOut = 64;    // output stage capacity (flushed at 32)
constexpr int kPQ = 40;     // warp queue of ionization products (built 32 at a time)
constexpr int kPQRow = 9;   // x y z, product speed, ax ay az of the ionizing electron, w, remaining time
constexpr int kAtt = 32;    // warp buffer of attachment events awaiting their deposit
template <class T> __device__ __forceinline__ int most_trips(const PushArgs<T>& A) {
    return sizeof(T) == 4 ? kTripsF32 : A.trip_limit;
}

template <class T> struct Stage {
    T in[32 * kRow];
    T out[kOut * kRow];
    uint64_t in_id[32], out_id[kOut];
    T pq[kPQ * kPQRow];
    uint64_t pq_id[kPQ];    // the ionizing electron
    uint32_t pq_k[kPQ];     // index of its draw that ionized
    T att[kAtt * 4];        // x y z w of negative-ion events
};

// Double precision: the electrons a warp has in flight (collide_pool).
constexpr int kPool = 64;
template <class T> struct Pool {
    T f[14][kPool];         // x, displacement, v, a (three each), w, remaining time
    T ht[kPool], hr[kPool]; // a hit's table coordinate and rate
    uint64_t id[kPool];
    uint32_t k[kPool], hz[kPool], hw[kPool];
    T out[kOut * kRow];
    uint64_t out_id[kOut];
    T pq[kPQ * kPQRow];
    uint64_t pq_id[kPQ];
    uint32_t pq_k[kPQ];
    T att[kAtt * 4];
    uint8_t draw[kPool], hit[kPool], idle[kPool];  // places whose next step is a draw, a collision; free ones
};
template <class T> struct WarpStage { typedef Stage<T> type; };
template <> struct WarpStage<double> { typedef Pool<double> type; };

template <class T> constexpr size_t collide_smem() {
    return ((sizeof(ProcSmem<T>) + 15) & ~(size_t)15) + 4 * sizeof(typename WarpStage<T>::type);
}

// Writes staged finished electrons [0, cnt) (lane l takes entry l): faces,
// electrode, output append, deposit or moments; then moves entries cnt..n-1 down.
template <class T, int MODE, class S>
__device__ __forceinline__ void flush_out(const PushArgs<T>& A, S* sg, int& n, int cnt, LStats& ls, MomAcc<T>& M) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    bool live = lane < cnt;
    T x[3], v[3], a[3], w = (T)0;
    uint64_t id = 0;
    if (live) {
        const T* r = sg->out + lane * kRow;
        x[0] = r[0]; x[1] = r[1]; x[2] = r[2];
        v[0] = r[3]; v[1] = r[4]; v[2] = r[5];
        a[0] = r[6]; a[1] = r[7]; a[2] = r[8];
        w = r[9];
        id = sg->out_id[lane];
        if (MODE == MODE_PIC) live = boundaries(A, x, v, w, ls);
    }
    const unsigned m = __ballot_sync(kFull, live);
    if (m) {
        unsigned long long s0 = 0;
        if (lane == 0) s0 = atomicAdd(&A.st->n_out, (unsigned long long)__popc(m));
        s0 = __shfl_sync(kFull, s0, 0);
        bool stored = false;
        if (live) {
            const unsigned long long slot = s0 + __popc(m & ((1u << lane) - 1u));
            if ((long long)slot < A.cap_out) {
                store(A.out, slot, x, v, a, w, id);
                stored = true;
                if (MODE == MODE_PIC) {
                    if (A.q_e) deposit_at(A, x[0], x[1], x[2], w, A.q_e);
                } else {
                    M.add(x, v, w);
                }
            } else {
                atomicOr(&A.st->err, kErrOutCapacity);
            }
        }
        if (MODE == MODE_PIC && A.vhist) {
            // the speed histogram of the time-step control (Sec. 2.1.4) over the stored electrons; lanes
            // with the same bin add once
            const int b = stored && w > (T)0 ? speed_bin((float)v[0], (float)v[1], (float)v[2]) : -1;
            const unsigned grp = __match_any_sync(kFull, b);
            if (b >= 0 && __ffs(grp) - 1 == lane) atomicAdd(&A.vhist[b], (unsigned)__popc(grp));
        }
    }
    __syncwarp();
    const int rest = n - cnt;
    if (lane < rest) {
        for (int f = 0; f < 10; ++f) sg->out[lane * kRow + f] = sg->out[(cnt + lane) * kRow + f];
        sg->out_id[lane] = sg->out_id[cnt + lane];
    }
    __syncwarp();
    n = rest;
}

// An ionization product as a work item of the input stage: derived id and
// direction from its own draw (make_child), its positive-ion event and, with
// photoionization, the photon test of the ionizing event (Sec. 2.4).  e: the
// compact entry (x y z, speed, a, w, remaining time) of electron pid's draw k.
template <class T, int MODE>
__device__ __forceinline__ void build_product(const PushArgs<T>& A, const T* e, uint64_t pid, uint32_t k, T* row,
                                              uint64_t* rid) {
    T vc[3];
    *rid = make_child(A.K, A.step, pid, k, e[3], vc);
    if (MODE == MODE_PIC) {
        if (A.q_pos) deposit_at(A, e[0], e[1], e[2], e[7], A.q_pos);
        if (A.photo_prob > (T)0) photo_test(A, A.K, A.step, pid, k, e, e[7]);
    }
    row[0] = e[0]; row[1] = e[1]; row[2] = e[2];
    row[3] = vc[0]; row[4] = vc[1]; row[5] = vc[2];
    row[6] = e[4]; row[7] = e[5]; row[8] = e[6];
    row[9] = e[7];
    row[10] = e[8];
}

// Deposits the buffered negative-ion events [0, n) of the warp, one per lane.
template <class T, class S> __device__ __forceinline__ void flush_att(const PushArgs<T>& A, S* sg, int& n) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < n) {
        const T* a = sg->att + lane * 4;
        deposit_at(A, a[0], a[1], a[2], a[3], A.q_neg);
    }
    __syncwarp();
    n = 0;
}

template <class T, int MODE, bool FAST, bool STATS, bool CHILD>
__device__ __forceinline__ void collide_loop(const PushArgs<T>& A, const ProcSmem<T>* ps, Stage<T>* sg) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long* cursor = CHILD ? &A.st->n_fetch_c : &A.st->n_fetch;
    const ChildQ<T>& src = (A.gen & 1) ? A.cq2 : A.cq;
    // products the warp queue cannot take: the parents' go to the queue of the
    // first children launch, a children launch's to the other queue
    const ChildQ<T>& dst = CHILD ? ((A.gen & 1) ? A.cq : A.cq2) : A.cq;
    unsigned long long* dst_cnt = CHILD ? ((A.gen & 1) ? &A.st->n_child : &A.st->n_spill) : &A.st->n_child;
    // work items of the launch (fixed while it runs; read again at each refill rather than held in registers)
    auto items = [&]() -> long long {
        if (!CHILD) return (long long)parent_items<MODE>(A.st);
        const long long n = (long long)((A.gen & 1) ? A.st->n_spill : A.st->n_child);
        return n < A.cap_child ? n : A.cap_child;
    };
    if (CHILD) {
        if (items() == 0) return;  // the warp queues took every product
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&A.st->n_updates, (unsigned long long)items());
    }
    LStats ls;
    ls.zero();
    MomAcc<T> M;
    if (MODE == MODE_SWARM) M.zero();
    const Rates<T> rates{A.table, A.nu_max, A.tau_scale};
    Lane<T> L;
    bool active = false, dry = false, first = true;
    // warp-uniform counters: input stage head and size, output stage size,
    // queued products, buffered negative-ion events
    int in_head = 0, in_count = 0, n_out = 0, n_pq = 0, n_att = 0, trips_left = most_trips(A);
    for (;;) {
        if (--trips_left < 0) { atomicOr(&A.st->err, kErrDraws); break; }
        // 1. idle lanes take staged work items
        const bool want = !active;
        const unsigned need = __ballot_sync(kFull, want);
        const int avail = in_count - in_head;
        if (need && avail > 0) {
            const int rank = __popc(need & lt);
            if (want && rank < avail) {
                const int e = in_head + rank;
                const T* r = sg->in + e * kRow;
                for (int d = 0; d < 3; ++d) { L.x[d] = r[d]; L.v[d] = r[3 + d]; L.a[d] = r[6 + d]; L.d[d] = (T)0; }
                L.w = r[9];
                L.t_left = r[10];
                L.id = sg->in_id[e];
                L.k = 1;
                active = L.w > (T)0;
                if (active) ++ls.processed;
            }
            const int took = __popc(need) < avail ? __popc(need) : avail;
            in_head += took;
        }
        // 2. refill the input stage once it is drained: 32 queued products when
        //    there are that many (the rest once the input has run dry), else 32
        //    work items of the input; every lane prepares one entry
        if (in_head >= in_count && (!dry || n_pq > 0)) {
            int cnt = 0;
            __syncwarp();
            if (n_pq >= 32 || (dry && n_pq > 0)) {
                cnt = n_pq < 32 ? n_pq : 32;
                if (lane < cnt) {
                    const int j = n_pq - cnt + lane;
                    build_product<T, MODE>(A, sg->pq + j * kPQRow, sg->pq_id[j], sg->pq_k[j], sg->in + lane * kRow,
                                           &sg->in_id[lane]);
                }
                if (lane == 0) atomicAdd(&A.st->n_updates, (unsigned long long)cnt);
                n_pq -= cnt;
            } else {
                // A warp's first items follow from its place, in an order that
                // fills the SMs and their four schedulers evenly; later ones
                // come from the cursor.  With few items a warp takes fewer at a
                // time, so that more schedulers work (a lane's chain of draws,
                // not the issue rate, takes the time then).  (Capacities are
                // below 2^31.)
                const unsigned warps = gridDim.x * (blockDim.x >> 5), n_items = (unsigned)items();
                unsigned chunk = 32;
                if (n_items <= 24u * warps) chunk = (n_items / warps + 8u) & ~7u;
                unsigned b = 0;
                if (first) {
                    b = ((((threadIdx.x >> 5) - blockIdx.x / (unsigned)A.sms) & 3u) * gridDim.x + blockIdx.x) * chunk;
                } else {
                    unsigned long long c = 0;
                    if (lane == 0) c = atomicAdd(cursor, (unsigned long long)chunk);
                    c = __shfl_sync(kFull, c, 0) + (unsigned long long)warps * chunk;
                    b = c < n_items ? (unsigned)c : n_items;
                }
                first = false;
                const int left = b < n_items ? (int)(n_items - b) : 0;
                if (left <= 0) {
                    dry = true;
                } else {
                    cnt = left < (int)chunk ? left : (int)chunk;
                    if (lane < cnt) {
                        const long long it = (long long)b + lane;
                        T* r = sg->in + lane * kRow;
                        if (CHILD) {
                            const Soa<T>& q = src.p;
                            const T e[kPQRow] = {q.r[PX][it], q.r[PY][it], q.r[PZ][it], q.r[VX][it], q.r[AX][it],
                                                 q.r[AY][it], q.r[AZ][it], q.r[PW][it], src.t_left[it]};
                            build_product<T, MODE>(A, e, q.id[it], src.k[it], r, &sg->in_id[lane]);
                        } else {
                            T f[10];
                            for (int q = 0; q < 10; ++q) f[q] = A.in.r[q][it];
                            if (MODE == MODE_SWARM) uniform_accel(A, f);
                            else half_kick(A, f);
                            for (int q = 0; q < 10; ++q) r[q] = f[q];
                            r[10] = A.dt;
                            sg->in_id[lane] = A.in.id[it];
                        }
                    }
                }
            }
            in_head = 0;
            in_count = cnt;
            trips_left = most_trips(A);
            __syncwarp();
        }
        // 3. termination
        if (!__any_sync(kFull, active)) {
            if (dry && in_head >= in_count && n_pq == 0) break;
            continue;
        }
        // 4. up to two draws, which halves the warp bookkeeping per draw
        T sp = (T)0;
        const int r = advance<T, MODE, FAST, STATS>(A, rates, A.K, A.step, ps, active, L, ls, sp);
        const bool done = r == EV_DONE, ion = r == EV_IONIZED, att = r == EV_ATTACHED;
        if (done || att) active = false;
        // 5. ionization products wait in the warp queue as compact entries (the
        //    queue of the next launch when it is full)
        const unsigned im = __ballot_sync(kFull, ion);
        if (im) {
            if (ion) {
                const int slot = n_pq + __popc(im & lt);
                const T e[kPQRow] = {L.x[0] + L.d[0], L.x[1] + L.d[1], L.x[2] + L.d[2], sp,
                                     L.a[0], L.a[1], L.a[2], L.w, L.t_left};
                if (slot < kPQ) {
                    T* q = sg->pq + slot * kPQRow;
                    for (int f = 0; f < kPQRow; ++f) q[f] = e[f];
                    sg->pq_id[slot] = L.id;
                    sg->pq_k[slot] = L.k - 1;
                    ++ls.children;
                } else {
                    const unsigned long long q = atomicAdd(dst_cnt, 1ull);
                    if ((long long)q < A.cap_child) {
                        const Soa<T>& d = dst.p;
                        d.r[PX][q] = e[0]; d.r[PY][q] = e[1]; d.r[PZ][q] = e[2];
                        d.r[VX][q] = sp;
                        d.r[AX][q] = e[4]; d.r[AY][q] = e[5]; d.r[AZ][q] = e[6];
                        d.r[PW][q] = L.w;
                        d.id[q] = L.id;
                        dst.t_left[q] = L.t_left;
                        dst.k[q] = L.k - 1;
                        ++ls.children;
                    } else {
                        atomicOr(&A.st->err, kErrChildCapacity);
                    }
                }
            }
            n_pq += __popc(im);
            if (n_pq > kPQ) n_pq = kPQ;
        }
        // 6. negative-ion events wait for a deposit by 32 lanes at once
        if (MODE == MODE_PIC) {
            const unsigned am = __ballot_sync(kFull, att);
            if (am && A.q_neg) {
                if (n_att + __popc(am) > kAtt) flush_att(A, sg, n_att);
                if (att) {
                    T* q = sg->att + (n_att + __popc(am & lt)) * 4;
                    q[0] = L.x[0] + L.d[0]; q[1] = L.x[1] + L.d[1]; q[2] = L.x[2] + L.d[2]; q[3] = L.w;
                }
                n_att += __popc(am);
            }
        }
        // 7. finished electrons
        const unsigned dm = __ballot_sync(kFull, done);
        if (dm) {
            if (done) {
                const int e = n_out + __popc(dm & lt);
                T* q = sg->out + e * kRow;
                q[0] = L.x[0] + L.d[0]; q[1] = L.x[1] + L.d[1]; q[2] = L.x[2] + L.d[2];
                q[3] = L.v[0]; q[4] = L.v[1]; q[5] = L.v[2];
                q[6] = L.a[0]; q[7] = L.a[1]; q[8] = L.a[2];
                q[9] = L.w;
                sg->out_id[e] = L.id;
            }
            n_out += __popc(dm);
            if (n_out >= 32) flush_out<T, MODE>(A, sg, n_out, 32, ls, M);
        }
    }
    if (n_out > 0) flush_out<T, MODE>(A, sg, n_out, n_out, ls, M);
    if (MODE == MODE_PIC && n_att > 0) flush_att(A, sg, n_att);
    if (STATS) flush_stats(A, ls, A.n_proc);
    if (MODE == MODE_SWARM) {
        M.m[14] += ls.w_ion;
        M.m[15] += ls.w_att;
        __syncthreads();
        flush_moments(A, M, reinterpret_cast<double*>(sg - (threadIdx.x >> 5)));  // block-wide scratch
    }
}

// The collision loop of double precision.  A warp operation costs the double
// pipe 18 clocks of the whole multiprocessor whatever its lanes, a draw about
// 1900 of them and a collision 2300, and six of ten draws are null collisions:
// a lane that owns an electron makes every warp pay for both at every draw.
// So a warp keeps up to 64 electrons in shared memory (moving one costs ~30
// shared accesses) and does, as long as there are enough, 32 draws or 32
// collisions at a time; places wait in lists.  A draw whose rate lies clearly
// above the interpolated total (by more than the two sums can differ) is a null
// collision at once; any other goes to the collision, which decides exactly.
// Same draws, same operations on each electron as collide_loop.  1e5 streamer
// electrons: 2.76 ms a step, a lane an electron 3.95; 1.4e4 swarm electrons,
// which hardly fill the warps: 197 and 190 us.
template <class T, int MODE, bool STATS, bool CHILD>
__device__ __forceinline__ void collide_pool(const PushArgs<T>& A, const ProcSmem<T>* ps, Pool<T>* sg) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long* cursor = CHILD ? &A.st->n_fetch_c : &A.st->n_fetch;
    const ChildQ<T>& src = (A.gen & 1) ? A.cq2 : A.cq;
    const ChildQ<T>& dst = CHILD ? ((A.gen & 1) ? A.cq : A.cq2) : A.cq;  // products the warp queue cannot take
    unsigned long long* dst_cnt = CHILD ? ((A.gen & 1) ? &A.st->n_child : &A.st->n_spill) : &A.st->n_child;
    long long items = (long long)(CHILD ? ((A.gen & 1) ? A.st->n_spill : A.st->n_child) : parent_items<MODE>(A.st));
    if (CHILD) {
        if (items > A.cap_child) items = A.cap_child;
        if (items == 0) return;
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&A.st->n_updates, (unsigned long long)items);
    }
    LStats ls;
    ls.zero();
    MomAcc<T> M;
    if (MODE == MODE_SWARM) M.zero();
    const Rates<T> rates{A.table, A.nu_max, A.tau_scale};
    // First items by place, one range a warp: as many warps on each SM as its
    // share fills with 32 electrons each (1.4e4 electrons, three warps an SM:
    // 197 us; two of 46 208, four of 23 210), then from the cursor.
    const unsigned n_items = (unsigned)items, sms = (unsigned)A.sms, warps = gridDim.x * (blockDim.x >> 5);
    const unsigned per_sm = (n_items + 32u * sms - 1) / (32u * sms);
    const unsigned chunk = per_sm > 0 ? (n_items + sms * per_sm - 1) / (sms * per_sm) : 1u;  // 32 at most
    unsigned next = ((((threadIdx.x >> 5) - blockIdx.x / sms) & 3u) * gridDim.x + blockIdx.x) * chunk;
    unsigned end = next < n_items ? (n_items - next < chunk ? n_items : next + chunk) : 0u;
    if (end == 0u) next = 0u;
    // warp-uniform: sizes of the lists, of the output stage, queued products, buffered negative-ion events
    int nd = 0, nh = 0, nf = kPool, n_out = 0, n_pq = 0, n_att = 0, trips_left = most_trips(A);
    bool dry = false;
    for (int q = lane; q < kPool; q += 32) sg->idle[q] = (uint8_t)q;
    for (;;) {
        if (--trips_left < 0) { atomicOr(&A.st->err, kErrDraws); break; }
        __syncwarp();
        const bool products = n_pq >= 32 || (dry && n_pq > 0);
        // 1. places are filled while fewer than 32 electrons wait for a draw
        if (nh < 32 && nd < 32 && (products || !dry) && (nf >= 8 || nd + nh == 0)) {
            int cnt = n_pq < 32 ? n_pq : 32;
            if (!products) {
                if (next >= end) {
                    unsigned long long c = 0;
                    if (lane == 0) c = atomicAdd(cursor, (unsigned long long)(nf < 32 ? nf : 32));
                    c = __shfl_sync(kFull, c, 0) + (unsigned long long)warps * chunk;
                    next = c < n_items ? (unsigned)c : n_items;
                    const unsigned most = (unsigned)(nf < 32 ? nf : 32);
                    end = n_items - next < most ? n_items : next + most;
                }
                cnt = (int)(end - next) < 32 ? (int)(end - next) : 32;
                if (cnt <= 0) {
                    dry = true;
                    continue;
                }
            }
            if (cnt > nf) cnt = nf;
            const bool on = lane < cnt;
            int p = 0;
            T r[kRow] = {};
            uint64_t id = 0;
            if (on) {
                p = sg->idle[nf - cnt + lane];
                if (products) {
                    const int j = n_pq - cnt + lane;
                    build_product<T, MODE>(A, sg->pq + j * kPQRow, sg->pq_id[j], sg->pq_k[j], r, &id);
                } else {
                    const long long it = (long long)next + lane;
                    if (CHILD) {
                        const Soa<T>& q = src.p;
                        const T e[kPQRow] = {q.r[PX][it], q.r[PY][it], q.r[PZ][it], q.r[VX][it], q.r[AX][it],
                                             q.r[AY][it], q.r[AZ][it], q.r[PW][it], src.t_left[it]};
                        build_product<T, MODE>(A, e, q.id[it], src.k[it], r, &id);
                    } else {
                        for (int q = 0; q < 10; ++q) r[q] = A.in.r[q][it];
                        if (MODE == MODE_SWARM) uniform_accel(A, r);
                        else half_kick(A, r);
                        r[10] = A.dt;
                        id = A.in.id[it];
                    }
                }
            }
            if (products) {
                if (lane == 0) atomicAdd(&A.st->n_updates, (unsigned long long)cnt);
                n_pq -= cnt;
            } else {
                next += (unsigned)cnt;
            }
            nf -= cnt;
            trips_left = most_trips(A);
            const bool alive = on && r[9] > (T)0;
            const unsigned am = __ballot_sync(kFull, alive), em = __ballot_sync(kFull, on && !alive);
            if (alive) {
                ++ls.processed;
                for (int q = 0; q < 3; ++q) {
                    sg->f[q][p] = r[q];
                    sg->f[3 + q][p] = (T)0;
                    sg->f[6 + q][p] = r[3 + q];
                    sg->f[9 + q][p] = r[6 + q];
                }
                sg->f[12][p] = r[9];
                sg->f[13][p] = r[10];
                sg->id[p] = id;
                sg->k[p] = 1;
                sg->draw[nd + __popc(am & lt)] = (uint8_t)p;
            }
            __syncwarp();
            if (on && !alive) sg->idle[nf + __popc(em & lt)] = (uint8_t)p;
            nd += __popc(am);
            nf += __popc(em);
            continue;
        }
        if (nd + nh == 0) break;  // nothing in flight, nothing to come
        Lane<T> L;
        Hit<T> h;
        int p = 0, r = EV_CONTINUE;
        T sp = (T)0;
        bool on;
        const bool draws = nh < 32 && nd >= nh;
        if (draws) {
            // 2. draws
            const int cnt = nd < 32 ? nd : 32;
            on = lane < cnt;
            nd -= cnt;
            if (on) {
                p = sg->draw[nd + lane];
                for (int q = 0; q < 3; ++q) { L.d[q] = sg->f[3 + q][p]; L.v[q] = sg->f[6 + q][p]; L.a[q] = sg->f[9 + q][p]; }
                L.t_left = sg->f[13][p];
                L.id = sg->id[p];
                L.k = sg->k[p];
                r = candidate<T, false>(A, rates, A.K, A.step, L, ls, h);
                if (r == EV_HIT) {
                    int j;
                    T f, t0, dt;
                    table_split(A, h.t, j, f);
                    LdTab<T>::pair(A.table + A.n_bins * kTableRow + 2 * j, t0, dt);
                    if (h.target >= (t0 + f * dt) * (T)(1.0 + 1e-12)) { ++ls.nulls; r = EV_CONTINUE; }
                }
                for (int q = 0; q < 3; ++q) { sg->f[3 + q][p] = L.d[q]; sg->f[6 + q][p] = L.v[q]; }
                sg->f[13][p] = L.t_left;
                sg->k[p] = L.k;
                if (r == EV_HIT) {
                    sg->ht[p] = h.t;
                    sg->hr[p] = h.target;
                    sg->hz[p] = h.z;
                    sg->hw[p] = h.w;
                }
            }
        } else {
            // 3. collisions
            const int cnt = nh < 32 ? nh : 32;
            on = lane < cnt;
            nh -= cnt;
            if (on) {
                p = sg->hit[nh + lane];
                for (int q = 0; q < 3; ++q) L.v[q] = sg->f[6 + q][p];
                L.w = sg->f[12][p];
                h.t = sg->ht[p];
                h.target = sg->hr[p];
                h.z = sg->hz[p];
                h.w = sg->hw[p];
                r = collide<T, MODE, STATS>(A, rates, ps, h, L, ls, sp);
                for (int q = 0; q < 3; ++q) sg->f[6 + q][p] = L.v[q];
            }
        }
        __syncwarp();
        const bool done = on && r == EV_DONE, ion = on && r == EV_IONIZED, att = on && r == EV_ATTACHED;
        // 4. back into the lists
        const unsigned cm = __ballot_sync(kFull, on && (r == EV_CONTINUE || ion)), hm = __ballot_sync(kFull, on && r == EV_HIT),
                       xm = __ballot_sync(kFull, done || att);
        if (cm >> lane & 1u) sg->draw[nd + __popc(cm & lt)] = (uint8_t)p;
        if (hm >> lane & 1u) sg->hit[nh + __popc(hm & lt)] = (uint8_t)p;
        if (xm >> lane & 1u) sg->idle[nf + __popc(xm & lt)] = (uint8_t)p;
        nd += __popc(cm);
        nh += __popc(hm);
        nf += __popc(xm);
        if (draws) {
            // 5. finished electrons
            const unsigned dm = __ballot_sync(kFull, done);
            if (dm) {
                if (done) {
                    const int e = n_out + __popc(dm & lt);
                    T* q = sg->out + e * kRow;
                    for (int d = 0; d < 3; ++d) {
                        q[d] = sg->f[d][p] + L.d[d];
                        q[3 + d] = L.v[d];
                        q[6 + d] = L.a[d];
                    }
                    q[9] = sg->f[12][p];
                    sg->out_id[e] = L.id;
                }
                n_out += __popc(dm);
                if (n_out >= 32) flush_out<T, MODE>(A, sg, n_out, 32, ls, M);
            }
            continue;
        }
        // 6. ionization products wait in the warp queue (the queue of the next launch when it is full)
        const unsigned im = __ballot_sync(kFull, ion);
        if (im) {
            if (ion) {
                const int slot = n_pq + __popc(im & lt);
                const T e[kPQRow] = {sg->f[0][p] + sg->f[3][p], sg->f[1][p] + sg->f[4][p], sg->f[2][p] + sg->f[5][p], sp,
                                     sg->f[9][p], sg->f[10][p], sg->f[11][p], L.w, sg->f[13][p]};
                const uint64_t id = sg->id[p];
                const uint32_t k = sg->k[p] - 1;
                if (slot < kPQ) {
                    T* q = sg->pq + slot * kPQRow;
                    for (int f = 0; f < kPQRow; ++f) q[f] = e[f];
                    sg->pq_id[slot] = id;
                    sg->pq_k[slot] = k;
                    ++ls.children;
                } else {
                    const unsigned long long q = atomicAdd(dst_cnt, 1ull);
                    if ((long long)q < A.cap_child) {
                        const Soa<T>& d = dst.p;
                        d.r[PX][q] = e[0]; d.r[PY][q] = e[1]; d.r[PZ][q] = e[2];
                        d.r[VX][q] = sp;
                        d.r[AX][q] = e[4]; d.r[AY][q] = e[5]; d.r[AZ][q] = e[6];
                        d.r[PW][q] = L.w;
                        d.id[q] = id;
                        dst.t_left[q] = e[8];
                        dst.k[q] = k;
                        ++ls.children;
                    } else {
                        atomicOr(&A.st->err, kErrChildCapacity);
                    }
                }
            }
            n_pq += __popc(im);
            if (n_pq > kPQ) n_pq = kPQ;
        }
        // 7. negative-ion events wait for a deposit by 32 lanes at once
        if (MODE == MODE_PIC) {
            const unsigned am = __ballot_sync(kFull, att);
            if (am && A.q_neg) {
                if (n_att + __popc(am) > kAtt) flush_att(A, sg, n_att);
                if (att) {
                    T* q = sg->att + (n_att + __popc(am & lt)) * 4;
                    for (int d = 0; d < 3; ++d) q[d] = sg->f[d][p] + sg->f[3 + d][p];
                    q[3] = L.w;
                }
                n_att += __popc(am);
            }
        }
    }
    if (n_out > 0) flush_out<T, MODE>(A, sg, n_out, n_out, ls, M);
    if (MODE == MODE_PIC && n_att > 0) flush_att(A, sg, n_att);
    if (STATS) flush_stats(A, ls, A.n_proc);
    if (MODE == MODE_SWARM) {
        M.m[14] += ls.w_ion;
        M.m[15] += ls.w_att;
        __syncthreads();
        flush_moments(A, M, reinterpret_cast<double*>(sg - (threadIdx.x >> 5)));  // block-wide scratch
    }
}

// Single precision keeps an electron on a lane; double precision pools them.
template <class T, int MODE, bool FAST, bool STATS, bool CHILD>
__device__ __forceinline__ void collide_items(const PushArgs<T>& A, const ProcSmem<T>* ps, typename WarpStage<T>::type* sg) {
    if constexpr (FAST) collide_loop<T, MODE, FAST, STATS, CHILD>(A, ps, sg);
    else collide_pool<T, MODE, STATS, CHILD>(A, ps, sg);
}

template <class T> __device__ __forceinline__ ProcSmem<T>* stage_proc(unsigned char* raw, const PushArgs<T>& A) {
    ProcSmem<T>* ps = reinterpret_cast<ProcSmem<T>*>(raw);
    if (threadIdx.x < 8) {
        ps->thr[threadIdx.x] = A.thr[threadIdx.x];
        ps->mratio[threadIdx.x] = A.mratio[threadIdx.x];
        ps->kind[threadIdx.x] = A.kind[threadIdx.x];
    }
    __syncthreads();
    return ps;
}

template <class T> __device__ __forceinline__ typename WarpStage<T>::type* warp_stage(unsigned char* raw) {
    typedef typename WarpStage<T>::type S;
    return reinterpret_cast<S*>(raw + ((sizeof(ProcSmem<T>) + 15) & ~(size_t)15)) + (threadIdx.x >> 5);
}

constexpr int kCollideThreads = 128;
// Resident blocks per SM the collision kernels are compiled for: six (24
// warps, 80 registers, 76 KB of L1 left beside their stages for the 40 KB of
// tables) in single precision, two in double precision (their double pipe is
// full then).  1e6 electrons in
// float: six 330 us, seven 356 (72 registers, 47 KB of L1), five 346.
template <class T> constexpr int collide_min_blocks() { return sizeof(T) == 4 ? 6 : 2; }

template <class T, int MODE, bool FAST, bool STATS>
__global__ void __launch_bounds__(kCollideThreads, collide_min_blocks<T>()) k_push(const PushArgs<T> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ProcSmem<T>* ps = stage_proc(smem_raw, A);
    collide_items<T, MODE, FAST, STATS, false>(A, ps, warp_stage<T>(smem_raw));
}

template <class T, int MODE, bool FAST, bool STATS>
__global__ void __launch_bounds__(kCollideThreads, collide_min_blocks<T>()) k_children(const PushArgs<T> A) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const ProcSmem<T>* ps = stage_proc(smem_raw, A);
    collide_items<T, MODE, FAST, STATS, true>(A, ps, warp_stage<T>(smem_raw));
}

// Deposit of the current particle set (no push).
template <class T>
__global__ void __launch_bounds__(256) k_deposit(const Soa<T> p, const DevState* st, T ox, T oy, T oz, T dx, int nx,
                                                 int ny, int nz, int axi, unsigned long long* q, DevState* stw) {
    const unsigned long long n = st->n_in;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (long long)n; i += stride) {
        const T w = p.r[PW][i];
        if (!(w > (T)0)) continue;
        const T x = p.r[PX][i], y = p.r[PY][i];
        if (axi) deposit(sqrt(x * x + y * y), oy + (T)0.5 * dx, p.r[PZ][i], w, ox, oy, oz, dx, nx, ny, nz, q, stw);
        else deposit(x, y, p.r[PZ][i], w, ox, oy, oz, dx, nx, ny, nz, q, stw);
    }
}

// Host-side launchers (defined in push_f32.cu / push_f64.cu).
template <class T> struct PushLaunch {
    static cudaError_t parents(const PushArgs<T>& A, int mode, bool stats, int grid, cudaStream_t s);
    static cudaError_t children(const PushArgs<T>& A, int mode, bool stats, int grid, cudaStream_t s);
    static cudaError_t deposit(const Soa<T>& p, DevState* st, const Grid& g, unsigned long long* q, int grid,
                               cudaStream_t s);
    static cudaError_t resample(const PushArgs<T>& A, int grid, cudaStream_t s);
    static cudaError_t photo_append(const PushArgs<T>& A, int grid, cudaStream_t s);
    static size_t smem_bytes(int n_bins);
    static int blocks_per_sm(int mode, int n_bins);
};

}  // namespace pic

// Transport-data surrogate: a 2 -> 128 -> 128 -> 6 network with tanh hidden
// units (the flux transport data of Sec. 2.2.4 as a function of log10 E/N and
// the O2 fraction), trained by full-batch Adam (Kingma & Ba 2015) on swarm
// results and evaluated on query points.
//
// The 128 x 128 layer is the only dense contraction: its forward product,
// the backpropagated product and the weight gradient run on the tensor cores
// in BF16 with FP32 accumulation (mma.sync m16n8k16).  The 2 -> 128 and
// 128 -> 6 layers, tanh, the loss and Adam run in FP32 on the CUDA cores.
// Reductions over points are per-block partial sums added in a fixed order
// (deterministic).
//
// Parameters (float32, one vector): W1[128][2], b1[128], W2[128][128], b2[128],
// W3[6][128], b3[6]; W[o][i] multiplies input i of unit o.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"
#include "graph_util.cuh"
#include "../../include/picmcc.h"

namespace mlp {

using pic::kFull;

constexpr int NI = MLP_NI, NH = MLP_NH, NO = MLP_NO;
constexpr int OFF_W1 = 0, OFF_B1 = NH * NI, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH, OFF_W3 = OFF_B2 + NH,
              OFF_B3 = OFF_W3 + NO * NH, NP = OFF_B3 + NO;
static_assert(NP == MLP_NPARAMS, "parameter count");

__device__ __forceinline__ float tanh_fast(float x) {
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// D = A B + C for one 16 x 8 x 16 tile (A row-major, B column-major, BF16
// inputs, FP32 accumulate).  Fragments: with g = lane / 4, t = lane % 4,
// a0 = A[g][2t, 2t+1], a1 = A[g+8][2t, 2t+1], a2 = A[g][2t+8, 2t+9],
// a3 = A[g+8][2t+8, 2t+9]; b0 = B[2t, 2t+1][g], b1 = B[2t+8, 2t+9][g];
// c0, c1 = C[g][2t, 2t+1], c2, c3 = C[g+8][2t, 2t+1].
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

constexpr long long kWaitLimit = 1ll << 26;
// Bounded wait for the barrier phase with the given parity; false on expiry.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    for (long long it = 0; it < kWaitLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// ------------------------------------------------------------------ training kernels
// BF16 copy of W2 ([o][i]).
__global__ void k_prep(const float* __restrict__ th, __nv_bfloat16* __restrict__ w2b) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < NH * NH) w2b[k] = __float2bfloat16_rn(th[OFF_W2 + k]);
}

// Forward and backward pass of kPts points in one block: nothing of it but
// the partial sums of the gradient leaves the chip.  The blocks of a split (up
// to 256 points, the depth of one accumulator of the weight gradient) form a
// cluster: every block copies its points' h1, and of dz2 the columns of their
// rows of gW2, into the others' shared memory as soon as they exist (bulk
// copies counted by the receiver's barrier: with 16-byte stores the two
// exchanges took 5000 of 24000 clocks, gathered by loads at the end 7000).
//
// What bounds it: the chain of dependent phases (loads, layer 1, two products,
// the head, its sums, the weight gradient; 600 to 2000 clocks each), one block
// an SM (220 KB), 16 warps.  64 points a block because that is the length of
// the partial sums.  4096 points: before, as six kernels with everything
// between them in global memory (transposed copies with 2-byte stores, sums
// read and written in shared memory), 51.9 us a step; now
// 13.3 (this kernel ~10).
constexpr int kPts = 64, kSplitPts = 256, kTrainThreads = 512, kHeadWarps = 8;
constexpr int kHeadPart = NO * NH + NO + NH + 1;  // partial sums of a block: gW3[6][128], gb3[6], gb2[128], loss
constexpr int kL1Part = NH * NI + NH;             // gW1[128][2], gb1[128]
constexpr int kBRow = NH + 8, kFRow = NH + 4;     // padded rows (16-byte pieces of eight rows on different banks)
// A cluster of `size` blocks: block r owns the 16-row tiles first(r) .. first(r + 1) - 1 of gW2.  dz2 is kept by
// owner, [owner][point][columns], rows of 16 BF16 a tile and 8 of padding.
__host__ __device__ constexpr int own_first(int r, int size) { return r * (NH / 16) / size; }
__host__ __device__ constexpr int own_row(int r, int size) { return (own_first(r + 1, size) - own_first(r, size)) * 16 + 8; }
constexpr int gd_size() {
    int most = 0;
    for (int size = 1; size <= kSplitPts / kPts; ++size)
        for (int r = 0; r < size; ++r) {
            const int n = size * kPts * own_row(r, size);
            most = n > most ? n : most;
        }
    return most;
}

__device__ __forceinline__ int owner_of(int tile, int size) {
    int r = 0;
    while (own_first(r + 1, size) <= tile) ++r;
    return r;
}
__device__ __forceinline__ int dz_base(int r, int size) { return kPts * (16 * own_first(r, size) + 8 * r); }

struct TrainSmem {
    __nv_bfloat16 gh[kSplitPts][kBRow], gd[gd_size()];  // h1 and dz2 of the split (the others write here)
    __nv_bfloat16 dzb[kPts * (NH + 8 * (kSplitPts / kPts))];
    union {
        __nv_bfloat16 w2[NH][kBRow];
        float part[kHeadWarps][kHeadPart + 1];  // once W2 is done with
    };
    float z[kPts][kFRow];  // z2, then h2, then dz1
    float h1[kPts][kFRow];
    float w3[NO * NH], dy[kPts][8], d[kPts][8], x[kPts][NI], tgt[kPts][NO];
    unsigned long long bar;
    int own_row[kSplitPts / kPts], own_base[kSplitPts / kPts];  // dzb by owner: columns a row, first element
    int tile_row[NH / 16], tile_base[NH / 16];                  // and by 16-column tile
};

// Four 8 x 8 BF16 matrices (TR: transposed); lane l gives the address of row
// l % 8 of matrix l / 8.
template <bool TR> __device__ __forceinline__ void ldm4(uint32_t (&r)[4], uint32_t a) {
    if (TR)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Copies bytes (a multiple of 16) from this block's shared address src to
// address dst of block `rank` of the cluster, whose barrier at bar counts them.
__device__ __forceinline__ void copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar, uint32_t rank) {
    uint32_t d, b;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(dst), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(bar), "r"(rank));
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(d),
                 "r"(src), "r"(bytes), "r"(b)
                 : "memory");
}

// acc += A B over K = 128 for a warp's 16 x 32 tile: A [m][k], the lane's
// address for 16-column step k given by a_at(k); B from column n0, as [n][k]
// or (BT) as [k][n]; k ascending, the operands of the next step loaded ahead.
template <bool BT, class F>
__device__ __forceinline__ void warp_tile(float (&acc)[4][4], F a_at, const __nv_bfloat16 (*B)[kBRow], int n0) {
    const int lane = threadIdx.x & 31, r8 = lane & 7, q = lane >> 3;
    uint32_t ba = BT ? smem_u32(&B[r8 + (q & 1) * 8][n0 + (q >> 1) * 8])
                     : smem_u32(&B[n0 + r8 + (q >> 1) * 8][(q & 1) * 8]);
    constexpr uint32_t kB = BT ? 16 * kBRow * 2 : 16 * 2, kH = BT ? 16 * 2 : 16 * kBRow * 2;
    uint32_t a[2][4], b[2][2][4];
    auto load = [&](int k) {
        ldm4<false>(a[k & 1], a_at(k));
        ldm4<BT>(b[k & 1][0], ba + k * kB);
        ldm4<BT>(b[k & 1][1], ba + k * kB + kH);
    };
    load(0);
#pragma unroll
    for (int k = 0; k < NH / 16; ++k) {
        const int s = k & 1;
        if (k + 1 < NH / 16) load(k + 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            mma_bf16(acc[2 * h], a[s][0], a[s][1], a[s][2], a[s][3], b[s][h][0], b[s][h][1]);
            mma_bf16(acc[2 * h + 1], a[s][0], a[s][1], a[s][2], a[s][3], b[s][h][2], b[s][h][3]);
        }
    }
}

// Sums over the lanes of 24 values, each by the butterfly 16, 8, 4, 2, 1 (lane
// l adds lane l ^ 16 first), the values halved between the partners on the
// way: the lane ends with the sum of value sum24_index(lane).
__device__ __forceinline__ float sum24(float (&v)[24], int lane) {
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        const float keep = lane & 16 ? v[12 + j] : v[j], give = lane & 16 ? v[j] : v[12 + j];
        v[j] = keep + __shfl_xor_sync(kFull, give, 16);
    }
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const float keep = lane & 8 ? v[6 + j] : v[j], give = lane & 8 ? v[j] : v[6 + j];
        v[j] = keep + __shfl_xor_sync(kFull, give, 8);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float keep = lane & 4 ? v[3 + j] : v[j], give = lane & 4 ? v[j] : v[3 + j];
        v[j] = keep + __shfl_xor_sync(kFull, give, 4);
    }
    v[3] = 0.0f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float keep = lane & 2 ? v[2 + j] : v[j], give = lane & 2 ? v[j] : v[2 + j];
        v[j] = keep + __shfl_xor_sync(kFull, give, 2);
    }
    const float keep = lane & 1 ? v[1] : v[0], give = lane & 1 ? v[0] : v[1];
    return keep + __shfl_xor_sync(kFull, give, 1);
}
__device__ __forceinline__ int sum24_index(int lane) {  // 24 and more: none
    const int low = lane & 3;
    return low == 3 ? 24 : (lane >> 4) * 12 + ((lane >> 3) & 1) * 6 + ((lane >> 2) & 1) * 3 + low;
}

// head: [block][kHeadPart], l1: [block][kL1Part], gw2: [cluster][128][128].
__global__ void __launch_bounds__(kTrainThreads, 1)
    k_backprop(const float* __restrict__ th, const __nv_bfloat16* __restrict__ w2b, const float* __restrict__ x,
               const float* __restrict__ tgt, float inv6n, float* __restrict__ head, float* __restrict__ l1,
               float* __restrict__ gw2) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int u = tid & (NH - 1), grp = tid >> 7;
    const int size = (int)cluster_size(), rank = (int)cluster_rank();
    const int own0 = own_first(rank, size), nt = own_first(rank + 1, size) - own0, row = own_row(rank, size);
    const size_t p0 = (size_t)blockIdx.x * kPts;
    __nv_bfloat16 (*h1b)[kBRow] = S.gh + rank * kPts;
    const uint32_t bar = smem_u32(&S.bar);
    if (tid == 0) {
        // one phase: h1 of the other blocks, dz2 of all
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        const uint32_t bytes = (size - 1) * sizeof(S.gh) / (kSplitPts / kPts) + size * kPts * row * 2;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
    }
    __syncwarp();
    cluster_arrive();  // (1) this block runs and its barrier stands
    // nothing of this depends on the kernel before
    if (tid >= 64 && tid < 64 + size) {
        S.own_row[tid - 64] = own_row(tid - 64, size);
        S.own_base[tid - 64] = dz_base(tid - 64, size);
    }
    if (tid >= 96 && tid < 96 + NH / 16) {
        const int k = tid - 96, r = owner_of(k, size);
        S.tile_row[k] = own_row(r, size);
        S.tile_base[k] = dz_base(r, size) + 16 * (k - own_first(r, size));
    }
    if (tid < kPts * NI) (&S.x[0][0])[tid] = x[p0 * NI + tid];
    if (tid < kPts * NO) (&S.tgt[0][0])[tid] = tgt[p0 * NO + tid];
    __syncthreads();
    pic::pdl_wait();
    cudaTriggerProgrammaticLaunchCompletion();
    const float w10 = th[OFF_W1 + u * NI], w11 = th[OFF_W1 + u * NI + 1], b1 = th[OFF_B1 + u];
    uint4 wv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) wv[j] = reinterpret_cast<const uint4*>(w2b)[tid + j * kTrainThreads];
    const float w3a = th[OFF_W3 + tid], w3b = tid < NO * NH - kTrainThreads ? th[OFF_W3 + kTrainThreads + tid] : 0.0f;
    float b2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) b2[q] = th[OFF_B2 + lane + 32 * q];
    const int si = sum24_index(lane);
    const float b3 = si < 24 ? th[OFF_B3 + si % NO] : 0.0f;
    // h1 = tanh(W1 x + b1)
#pragma unroll 4
    for (int p = grp; p < kPts; p += kTrainThreads / NH) {
        const float h = tanh_fast(fmaf(w11, S.x[p][1], fmaf(w10, S.x[p][0], b1)));
        S.h1[p][u] = h;
        h1b[p][u] = __float2bfloat16_rn(h);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int q = tid + j * kTrainThreads;  // 16 pieces a row
        *reinterpret_cast<uint4*>(&S.w2[q >> 4][(q & 15) * 8]) = wv[j];
    }
    S.w3[tid] = w3a;
    if (tid < NO * NH - kTrainThreads) S.w3[kTrainThreads + tid] = w3b;
    fence_async_smem();
    __syncthreads();
    cluster_wait();  // (1)
    if (tid < size && tid != rank)
        copy_to_peer(smem_u32(h1b), smem_u32(h1b), sizeof(S.gh) / (kSplitPts / kPts), bar, tid);
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32, g = lane >> 2, t = lane & 3;
    {
        float acc[4][4] = {};
        const uint32_t a0 = smem_u32(&h1b[m0 + (lane & 15)][(lane >> 4) * 8]);
        warp_tile<false>(acc, [&](int k) { return a0 + k * 32; }, S.w2, n0);  // z2 = h1 W2^T
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            *reinterpret_cast<float2*>(&S.z[m0 + g][n0 + 8 * j + 2 * t]) = make_float2(acc[j][0], acc[j][1]);
            *reinterpret_cast<float2*>(&S.z[m0 + g + 8][n0 + 8 * j + 2 * t]) = make_float2(acc[j][2], acc[j][3]);
        }
    }
    __syncthreads();
    // output layer: a warp takes four points, a lane units lane, lane + 32, ...
    {
        float y[24], w3[NO][4];
#pragma unroll
        for (int o = 0; o < NO; ++o)
#pragma unroll
            for (int q = 0; q < 4; ++q) w3[o][q] = S.w3[o * NH + lane + 32 * q];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float h2[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float* zp = &S.z[warp * 4 + j][lane + 32 * q];
                h2[q] = tanh_fast(*zp + b2[q]);
                *zp = h2[q];
            }
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                float s = 0.0f;
#pragma unroll
                for (int q = 0; q < 4; ++q) s = fmaf(w3[o][q], h2[q], s);
                y[j * NO + o] = s;
            }
        }
        const float yo = sum24(y, lane) + b3;
        if (si < 24) {
            const int p = warp * 4 + si / NO, o = si % NO;
            const float d = yo - S.tgt[p][o];
            S.d[p][o] = d;
            S.dy[p][o] = 2.0f * d * inv6n;
        }
    }
    __syncthreads();
    // dz2 and the sums over the points: eight chains (points w, w + 8, ...), kept for the sum of the eight in order
    float acc3[2][NO], gb2[2];
    {
        float w3[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) w3[o] = S.w3[o * NH + u];
        const int dzr = S.tile_row[u / 16];
        __nv_bfloat16* dzc = S.dzb + S.tile_base[u / 16] + u % 16;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
#pragma unroll
            for (int o = 0; o < NO; ++o) acc3[v][o] = 0.0f;
            gb2[v] = 0.0f;
        }
#pragma unroll 2
        for (int c = 0; c < kPts / kHeadWarps; ++c)
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const int p = 2 * grp + v + c * kHeadWarps;
                const float h2 = S.z[p][u];
                const float4 da = *reinterpret_cast<const float4*>(&S.dy[p][0]);
                const float2 db = *reinterpret_cast<const float2*>(&S.dy[p][4]);
                const float dy[NO] = {da.x, da.y, da.z, da.w, db.x, db.y};
                float dh = 0.0f;
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    acc3[v][o] = fmaf(dy[o], h2, acc3[v][o]);
                    dh = fmaf(w3[o], dy[o], dh);
                }
                const float dz = __fmul_rn(dh, fmaf(-h2, h2, 1.0f));
                gb2[v] = __fadd_rn(gb2[v], dz);
                dzc[p * dzr] = __float2bfloat16_rn(dz);
            }
    }
    fence_async_smem();
    __syncthreads();
    // dz2 to the owners of its columns
    if (tid < size) {
        const int to = S.own_row[tid];
        copy_to_peer(smem_u32(&S.gd[rank * kPts * to]), smem_u32(&S.dzb[S.own_base[tid]]), kPts * to * 2, bar, tid);
    }
    {
        float acc[4][4] = {};
        const uint32_t a0 = smem_u32(&S.dzb[(lane >> 4) * 8]);
        const int pr = m0 + (lane & 15);
        warp_tile<true>(acc, [&](int k) { return a0 + 2 * (S.tile_base[k] + pr * S.tile_row[k]); },  // dh1 = dz2 W2
                        S.w2, n0);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {  // dz1 = dh1 (1 - h1^2)
                const int p = m0 + g + 8 * h, i = n0 + 8 * j + 2 * t;
                const float2 h1 = *reinterpret_cast<const float2*>(&S.h1[p][i]);
                *reinterpret_cast<float2*>(&S.z[p][i]) =
                    make_float2(__fmul_rn(acc[j][2 * h], fmaf(-h1.x, h1.x, 1.0f)),
                                __fmul_rn(acc[j][2 * h + 1], fmaf(-h1.y, h1.y, 1.0f)));
            }
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 2; ++v) {
#pragma unroll
        for (int o = 0; o < NO; ++o) S.part[2 * grp + v][o * NH + u] = acc3[v][o];
        S.part[2 * grp + v][NO * NH + NO + u] = gb2[v];
    }
    if (tid < kHeadWarps * (NO + 1)) {
        const int w = tid / (NO + 1), o = tid % (NO + 1);
        float s = 0.0f;
        for (int p = w; p < kPts; p += kHeadWarps) {
            if (o < NO) {
                s += S.dy[p][o];
            } else {
                float l = 0.0f;
                for (int q = 0; q < NO; ++q) l = fmaf(S.d[p][q], S.d[p][q], l);
                s += l;
            }
        }
        S.part[w][o < NO ? NO * NH + o : kHeadPart - 1] = s;
    }
    // sums of dz1 over the points, in order
    if (grp == 3) {
        float g0 = 0.0f, g1 = 0.0f, gb = 0.0f;
#pragma unroll 8
        for (int p = 0; p < kPts; ++p) {
            const float dz = S.z[p][u];
            const float2 xp = *reinterpret_cast<const float2*>(&S.x[p][0]);
            g0 = fmaf(dz, xp.x, g0);
            g1 = fmaf(dz, xp.y, g1);
            gb += dz;
        }
        float* out = l1 + (size_t)blockIdx.x * kL1Part;
        out[u * NI] = g0;
        out[u * NI + 1] = g1;
        out[NH * NI + u] = gb;
    }
    __syncthreads();
#pragma unroll 1
    for (int k = tid; k < kHeadPart; k += kTrainThreads) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < kHeadWarps; ++w) s += S.part[w][k];
        head[(size_t)blockIdx.x * kHeadPart + k] = s;
    }
    const bool got = bar_wait(bar, 0);
    __syncwarp();
    cluster_arrive();  // (2) what this block was sent has arrived
    // gW2 = dz2^T h1 over the split's points, in order: this block's 16-row tiles
    const int pts = got ? size * kPts : 0;
    float* out = gw2 + ((size_t)(blockIdx.x / size) * NH + own0 * 16) * NH;
    // a warp takes 16 columns of two row tiles (half the warps of 32 x 16: 1536 clocks of shared-memory reads
    // in place of 2048)
    const int r8 = lane & 7, q4 = lane >> 3;
#pragma unroll 1
    for (int it = warp; it < (nt + 1) / 2 * 8; it += kTrainThreads / 32) {
        const int o0 = (it >> 3) * 32, i0 = (it & 7) * 16;
        const bool two = o0 + 16 < nt * 16;
        uint32_t aa = smem_u32(&S.gd[(r8 + (q4 >> 1) * 8) * row + o0 + (q4 & 1) * 8]);
        uint32_t ba = smem_u32(&S.gh[r8 + (q4 & 1) * 8][i0 + (q4 >> 1) * 8]);
        const uint32_t a2 = two ? 32 : 0;
        float acc[4][4] = {};
        if (!got) acc[0][0] = __int_as_float(0x7fc00000);  // the wait expired: no gradient
#pragma unroll 1
        for (int k = 0; k < pts; k += 64) {
            uint32_t a[4][2][4], b[4][4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                ldm4<true>(a[s][0], aa);
                ldm4<true>(b[s], ba);
                ldm4<true>(a[s][1], aa + a2);
                aa += 16 * row * 2;
                ba += 16 * kBRow * 2;
            }
#pragma unroll
            for (int s = 0; s < 4; ++s)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    mma_bf16(acc[2 * h], a[s][h][0], a[s][h][1], a[s][h][2], a[s][h][3], b[s][0], b[s][1]);
                    mma_bf16(acc[2 * h + 1], a[s][h][0], a[s][h][1], a[s][h][2], a[s][h][3], b[s][2], b[s][3]);
                }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = o0 + (j >> 1) * 16 + g, c = i0 + 8 * (j & 1) + 2 * t;
            if (j >= 2 && !two) break;
            *reinterpret_cast<float2*>(out + r * NH + c) = make_float2(acc[j][0], acc[j][1]);
            *reinterpret_cast<float2*>(out + (r + 8) * NH + c) = make_float2(acc[j][2], acc[j][3]);
        }
    }
    __syncwarp();
    cluster_wait();  // (2) this block's memory has been read
}

struct Parts {
    const float* gw2;   // [splits][128][128]
    const float* head;  // [n_head][kHeadPart]
    const float* l1;    // [n_l1][kL1Part]
    int splits, n_head, n_l1;
};

// Sum of n values `stride` apart, in order, 64 loads in flight.
__device__ __forceinline__ float sum_rows(const float* __restrict__ p, size_t stride, int n) {
    float s = 0.0f;
    for (; n >= 64; n -= 64) {
        float v[64];
#pragma unroll
        for (int q = 0; q < 64; ++q, p += stride) v[q] = *p;
#pragma unroll
        for (int q = 0; q < 64; ++q) s += v[q];
    }
#pragma unroll 16
    for (; n > 0; --n, p += stride) s += *p;
    return s;
}

// Gradient of parameter k from the partial sums, added in a fixed order.
__device__ __forceinline__ float grad_of(const Parts& P, int k) {
    // W1 then b1, b2, W3, b3: places in the rows of partial sums
    if (k < OFF_W2) return sum_rows(P.l1 + k, kL1Part, P.n_l1);
    if (k < OFF_B2) return sum_rows(P.gw2 + (k - OFF_W2), NH * NH, P.splits);
    const int j = k < OFF_W3 ? NO * NH + NO + (k - OFF_B2) : (k < OFF_B3 ? k - OFF_W3 : NO * NH + (k - OFF_B3));
    return sum_rows(P.head + j, kHeadPart, P.n_head);
}

__device__ __forceinline__ void write_loss(const Parts& P, float* loss, float inv6n) {
    if (loss) *loss = sum_rows(P.head + kHeadPart - 1, kHeadPart, P.n_head) * inv6n;
}
// A thread beyond the parameters (of another warp) adds the loss.
constexpr int kParamThreads = 128, kParamBlocks = NP / kParamThreads + 1, kLossThread = kParamBlocks * kParamThreads - 1;
static_assert(kLossThread >= NP, "a thread for the loss");

__global__ void k_grad_out(Parts P, float* __restrict__ grad, float* __restrict__ loss, float inv6n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < NP) grad[k] = grad_of(P, k);
    if (k == kLossThread) write_loss(P, loss, inv6n);
}

// Adam (Kingma & Ba 2015, Algorithm 1), step `step` (from 1), on every
// parameter, then the BF16 copy of W2 for the next step.  One round trip for
// up to 64 rows of partial sums, which the rest hides behind; the loss on a warp
// of its own.  4096 points: ~3 us behind the kernel before (6.3 with dependent
// loads and a kernel that counted the steps).
__global__ void __launch_bounds__(kParamThreads) k_adam(Parts P, float* __restrict__ th, float* __restrict__ m,
                                                        float* __restrict__ v, int step, float lr, float beta1,
                                                        float beta2, float eps, __nv_bfloat16* __restrict__ w2b,
                                                        float* __restrict__ loss, float inv6n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
    pic::pdl_wait();
    cudaTriggerProgrammaticLaunchCompletion();
    if (k < NP) {
        const float m0 = m[k], v0 = v[k], t0 = th[k];
        const float gk = grad_of(P, k);
        const float mk = fmaf(1.0f - beta1, gk, beta1 * m0);
        const float vk = fmaf((1.0f - beta2) * gk, gk, beta2 * v0);
        m[k] = mk;
        v[k] = vk;
        const float nt = t0 - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
        th[k] = nt;
        if (k >= OFF_W2 && k < OFF_B2) w2b[k - OFF_W2] = __float2bfloat16_rn(nt);
    }
    if (k == kLossThread) write_loss(P, loss, inv6n);
}

// ------------------------------------------------------------------ inference
// Fused forward pass.  Four warps per block; each warp takes 16 points at a
// time: layer 1 on the CUDA cores into a BF16 tile in shared memory, the
// 128 x 128 layer by mma.sync against W2 (BF16, resident in shared memory),
// tanh and the 128 -> 6 layer in the accumulator registers, reduced over the
// four lanes that share a row.
constexpr int kInfWarps = 4, kRowPad = NH + 8;
struct InfSmem {
    __nv_bfloat16 w2[NH][kRowPad];
    __nv_bfloat16 h1[kInfWarps][16][kRowPad];
    float w1[NH * NI], b1[NH], b2[NH], w3[NO * NH], b3[NO];
};

__global__ void __launch_bounds__(kInfWarps * 32) k_infer(const float* __restrict__ th,
                                                          const __nv_bfloat16* __restrict__ w2b,
                                                          const float* __restrict__ x, float* __restrict__ y,
                                                          long long n) {
    extern __shared__ __align__(16) unsigned char inf_raw[];
    InfSmem& S = *reinterpret_cast<InfSmem*>(inf_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    for (int k = tid; k < NH * NH / 2; k += blockDim.x) {
        const int o = (2 * k) / NH, i = (2 * k) % NH;
        *reinterpret_cast<uint32_t*>(&S.w2[o][i]) = reinterpret_cast<const uint32_t*>(w2b)[k];
    }
    for (int k = tid; k < NH * NI; k += blockDim.x) S.w1[k] = th[OFF_W1 + k];
    for (int k = tid; k < NH; k += blockDim.x) {
        S.b1[k] = th[OFF_B1 + k];
        S.b2[k] = th[OFF_B2 + k];
    }
    for (int k = tid; k < NO * NH; k += blockDim.x) S.w3[k] = th[OFF_W3 + k];
    if (tid < NO) S.b3[tid] = th[OFF_B3 + tid];
    __syncthreads();
    const long long n_tiles = (n + 15) / 16;
    for (long long tile = (long long)blockIdx.x * kInfWarps + warp; tile < n_tiles;
         tile += (long long)gridDim.x * kInfWarps) {
        const long long p0 = tile * 16;
        // inputs of the 16 points (lanes 0..15 load, everyone reads by shuffle)
        float x0 = 0.0f, x1 = 0.0f;
        if (lane < 16 && p0 + lane < n) {
            x0 = x[(p0 + lane) * NI];
            x1 = x[(p0 + lane) * NI + 1];
        }
        // layer 1: lane covers units lane + 32 q for all 16 points
#pragma unroll 4
        for (int r = 0; r < 16; ++r) {
            const float a0 = __shfl_sync(kFull, x0, r), a1 = __shfl_sync(kFull, x1, r);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int u = lane + 32 * q;
                const float z = fmaf(S.w1[u * NI + 1], a1, fmaf(S.w1[u * NI], a0, S.b1[u]));
                S.h1[warp][r][u] = __float2bfloat16_rn(tanh_fast(z));
            }
        }
        __syncwarp();
        // layer 2 on the tensor cores: acc[nt] covers output units 8 nt .. 8 nt + 7
        float acc[NH / 8][4];
#pragma unroll
        for (int nt = 0; nt < NH / 8; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.0f;
#pragma unroll
        for (int kk = 0; kk < NH; kk += 16) {
            const uint32_t a0 = *reinterpret_cast<const uint32_t*>(&S.h1[warp][g][kk + 2 * t]);
            const uint32_t a1 = *reinterpret_cast<const uint32_t*>(&S.h1[warp][g + 8][kk + 2 * t]);
            const uint32_t a2 = *reinterpret_cast<const uint32_t*>(&S.h1[warp][g][kk + 2 * t + 8]);
            const uint32_t a3 = *reinterpret_cast<const uint32_t*>(&S.h1[warp][g + 8][kk + 2 * t + 8]);
#pragma unroll
            for (int nt = 0; nt < NH / 8; ++nt) {
                const uint32_t b0 = *reinterpret_cast<const uint32_t*>(&S.w2[nt * 8 + g][kk + 2 * t]);
                const uint32_t b1 = *reinterpret_cast<const uint32_t*>(&S.w2[nt * 8 + g][kk + 2 * t + 8]);
                mma_bf16(acc[nt], a0, a1, a2, a3, b0, b1);
            }
        }
        __syncwarp();
        // tanh and the output layer for rows g and g + 8
        float ya[NO], yb[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) ya[o] = yb[o] = 0.0f;
#pragma unroll
        for (int nt = 0; nt < NH / 8; ++nt) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int u = nt * 8 + 2 * t + e;
                const float ha = tanh_fast(acc[nt][e] + S.b2[u]);
                const float hb = tanh_fast(acc[nt][2 + e] + S.b2[u]);
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    ya[o] = fmaf(S.w3[o * NH + u], ha, ya[o]);
                    yb[o] = fmaf(S.w3[o * NH + u], hb, yb[o]);
                }
            }
        }
#pragma unroll
        for (int o = 0; o < NO; ++o) {
            ya[o] += __shfl_xor_sync(kFull, ya[o], 1);
            ya[o] += __shfl_xor_sync(kFull, ya[o], 2);
            yb[o] += __shfl_xor_sync(kFull, yb[o], 1);
            yb[o] += __shfl_xor_sync(kFull, yb[o], 2);
        }
        if (t == 0) {
            const long long pa = p0 + g, pb = p0 + g + 8;
            if (pa < n)
#pragma unroll
                for (int o = 0; o < NO; ++o) y[pa * NO + o] = ya[o] + S.b3[o];
            if (pb < n)
#pragma unroll
                for (int o = 0; o < NO; ++o) y[pb * NO + o] = yb[o] + S.b3[o];
        }
    }
}

// ------------------------------------------------------------------ inference on tcgen05
// Fused forward pass on the fifth-generation tensor cores.  A block holds W2
// once and has four groups of 256 threads; a group takes 128 points at a time:
//   1. layer 1 in FP32 (thread: eight units of every 16th point, the units'
//      weights in registers), tanh in packed BF16, written as the A operand
//      (128 points x 128 units) in shared memory;
//   2. one thread issues eight 128 x 128 x 16 MMAs (A: h1, B: W2 resident in
//      shared memory) into a 128-column FP32 accumulator in tensor memory;
//   3. the accumulator rows are read back (row = point = TMEM lane; thread t:
//      point t % 128, units 64 (t / 128) on), bias and tanh applied, and h2
//      written over the A operand;
//   4. eight 128 x 16 x 16 MMAs against W3 (padded to 16 outputs) into the
//      first 16 accumulator columns; the first half of the threads read the
//      six outputs back, add b3 and store.
//
// What bounds it: the tanh unit (16 clocks of a scheduler for a packed pair a
// lane, measured: 2048 of a tile's 2530 clocks on a multiprocessor).  A group
// alone would leave it idle for two thirds of a tile (both products and their
// waits), so the four run independently of one another, each with its own
// named barrier, A operand and 128 of the 512 tensor-memory columns.  16.8
// million points: three blocks of one group an SM, a thread's weights loaded
// as broadcasts (63 % of the shared-memory pipe) 1323 us; weights by unit 1286;
// four groups in a block 1156.  Layer 1 of the next tile during the waits
// (held in registers, which then spill): 1188.
// Operands use the canonical K-major layout without swizzle: core matrices
// of 8 rows x 16 bytes stored contiguously, the next core matrix along K at
// +128 bytes, the next 8-row group at +2048 bytes (the same strides for the
// 16-row W3 tile, 4 KB).  Every MMA reads at most start + 15 x 2048 + 255
// bytes, inside its 32 KB (4 KB) tile.  Waits on the MMA completion barrier are
// bounded; on expiry the block writes NaN outputs, records the error and
// leaves, releasing its tensor memory.
constexpr int kTcGroups = 4, kTcGroup = 256, kTcThreads = kTcGroups * kTcGroup, kTcRows = 128;
constexpr uint32_t kTile = kTcRows * NH * 2;   // one 128 x 128 BF16 operand: 32 KB
constexpr uint32_t kLbo = 128, kSbo = 2048;    // core-matrix strides (bytes) along K and along M/N
constexpr uint32_t kB2Bytes = 16 * NH * 2;     // W3 padded to 16 rows: 4 KB

struct TcSmem {
    alignas(1024) unsigned char w2[kTile];   // B of layer 2: row o (output unit), K = input unit
    alignas(1024) unsigned char a[kTcGroups][kTile];  // A of a group: row = point, K = unit (h1, then h2)
    alignas(1024) unsigned char w3[kB2Bytes];
    alignas(16) float w1a[NH], w1b[NH], b1[NH], b2[NH];  // w1a, w1b: weights of the two inputs
    float2 xs[kTcGroups][2][kTcRows];                    // inputs of this tile and the next
    float b3[NO];
    alignas(8) unsigned long long bar[kTcGroups];
    uint32_t tmem;
    int abort[kTcGroups];
};

// byte offset of element (row r, k) in a K-major no-swizzle operand
__host__ __device__ constexpr uint32_t kmajor_off(uint32_t r, uint32_t k) {
    return (r >> 3) * kSbo + (k >> 3) * kLbo + (r & 7) * 16 + (k & 7) * 2;
}

// Shared-memory matrix descriptor: start address, leading (K) and stride
// (M/N) byte offsets in 16-byte units, the fixed version bits 46-47 = 1,
// no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16
// A and B (bits 7-9 = 1, 10-12 = 1), both K-major, N / 8 in bits 17-22,
// M / 16 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(uint32_t m, uint32_t n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
        "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __uint_as_float(r[q]);
}

// Pairs of floats in a 64-bit register, and the packed operations on them
// (each half rounded as the scalar operation).
__device__ __forceinline__ uint64_t pair_of(float lo, float hi) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t v;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
    return v;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t v;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
    return v;
}
__device__ __forceinline__ void ld_pairs(const float* p, uint64_t& a, uint64_t& b) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    a = v.x;
    b = v.y;
}

// tanh of a pair as packed BF16 (hardware approximation)
__device__ __forceinline__ uint32_t tanh_bf16x2(uint64_t v) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    uint32_t in = pack_bf16(lo, hi), out;
    asm("tanh.approx.bf16x2 %0, %1;" : "=r"(out) : "r"(in));
    return out;
}

__global__ void __launch_bounds__(kTcThreads, 1) k_infer_tc(const float* __restrict__ th,
                                                         const __nv_bfloat16* __restrict__ w2b,
                                                         const float* __restrict__ x, float* __restrict__ y,
                                                         long long n, int* __restrict__ err) {
    extern __shared__ __align__(1024) unsigned char tc_raw[];
    // align the operand tiles to 1024 bytes
    TcSmem& S = *reinterpret_cast<TcSmem*>(tc_raw + ((1024 - (smem_u32(tc_raw) & 1023)) & 1023));
    const int tid = threadIdx.x, warp = tid >> 5;
    const int group = tid / kTcGroup, gt = tid % kTcGroup, row = gt & (kTcRows - 1), half = gt >> 7;
    // operands and parameters
    for (int q = tid; q < NH * NH / 8; q += kTcThreads)  // eight inputs of a unit are 16 bytes in both layouts
        *reinterpret_cast<uint4*>(S.w2 + kmajor_off(q / (NH / 8), q % (NH / 8) * 8)) =
            reinterpret_cast<const uint4*>(w2b)[q];
    for (int k = tid; k < 16 * NH; k += kTcThreads) {
        const int o = k / NH, i = k % NH;
        *reinterpret_cast<__nv_bfloat16*>(S.w3 + kmajor_off(o, i)) =
            __float2bfloat16_rn(o < NO ? th[OFF_W3 + o * NH + i] : 0.0f);
    }
    for (int k = tid; k < NH; k += kTcThreads) {
        S.w1a[k] = th[OFF_W1 + k * NI];
        S.w1b[k] = th[OFF_W1 + k * NI + 1];
        S.b1[k] = th[OFF_B1 + k];
        S.b2[k] = th[OFF_B2 + k];
    }
    if (tid < NO) S.b3[tid] = th[OFF_B3 + tid];
    const auto x_of = [&](long long p) { return p < n ? make_float2(x[p * NI], x[p * NI + 1]) : make_float2(0.0f, 0.0f); };
    const long long first = blockIdx.x + (long long)gridDim.x * group, stride = (long long)gridDim.x * kTcGroups;
    if (half == 0) S.xs[group][0][row] = x_of(first * kTcRows + row);
    const uint32_t bar = smem_u32(&S.bar[group]);
    if (gt == 0) {
        S.abort[group] = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&S.tmem)),
                     "r"(128 * kTcGroups)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem + 128u * group;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t a_addr = smem_u32(S.a[group]), w2_addr = smem_u32(S.w2), w3_addr = smem_u32(S.w3);
    uint32_t parity = 0;
    const long long n_tiles = (n + kTcRows - 1) / kTcRows;
    // layer 1: units u1 .. u1 + 7 of rows r1, r1 + 16, ...
    const int lane = tid & 31, u1 = ((lane >> 3) + 4 * (warp & 3)) * 8, r1 = (lane & 7) + 8 * ((warp >> 2) & 1);
    unsigned char* const A = S.a[group];
    const auto sync = [&]() { pic::bar_named(1 + group, kTcGroup); };
    int buf = 0;
    for (long long tile = first; tile < n_tiles; tile += stride, buf ^= 1) {
        const long long p = tile * kTcRows + row;
        const bool valid = p < n;
        // the next tile's inputs, loaded one tile ahead
        float2 xn = make_float2(0.0f, 0.0f);
        if (half == 0) xn = x_of((tile + stride) * kTcRows + row);
        // 1. layer 1 into the A operand
        {
            uint64_t wa[4], wb[4], bb[4];
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                ld_pairs(&S.w1a[u1 + 2 * e], wa[e], wa[e + 1]);
                ld_pairs(&S.w1b[u1 + 2 * e], wb[e], wb[e + 1]);
                ld_pairs(&S.b1[u1 + 2 * e], bb[e], bb[e + 1]);
            }
#pragma unroll
            for (int j = 0; j < kTcRows / 16; ++j) {
                const float2 xr = S.xs[group][buf][r1 + 16 * j];
                const uint64_t x0 = pair_of(xr.x, xr.x), x1 = pair_of(xr.y, xr.y);
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) w[e] = tanh_bf16x2(fma2(wb[e], x1, fma2(wa[e], x0, bb[e])));
                *reinterpret_cast<uint4*>(A + kmajor_off(r1 + 16 * j, u1)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        if (half == 0) S.xs[group][buf ^ 1][row] = xn;
        fence_async_smem();
        sync();
        // 2. h1 W2^T into the accumulator
        if (gt == 0) {
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < NH / 16; ++kk)
                tc_mma(tmem, sdesc(a_addr + kk * 2 * kLbo, kLbo, kSbo), sdesc(w2_addr + kk * 2 * kLbo, kLbo, kSbo),
                       idesc_bf16(128, 128), kk > 0 ? 1u : 0u);
            tc_commit(bar);
        }
        if (!bar_wait(bar, parity)) S.abort[group] = 1;
        parity ^= 1;
        tc_fence_after();
        sync();
        if (S.abort[group]) break;
        // 3. bias, tanh, h2 over the A operand
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
            const int c0 = half * 64 + ch * 32;
            float acc[32];
            tmem_ld32(tmem + lane_base + (uint32_t)c0, acc);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                    const int q = c * 8 + 2 * e;
                    uint64_t b0, b1;
                    ld_pairs(&S.b2[c0 + q], b0, b1);
                    w[e] = tanh_bf16x2(add2(pair_of(acc[q], acc[q + 1]), b0));
                    w[e + 1] = tanh_bf16x2(add2(pair_of(acc[q + 2], acc[q + 3]), b1));
                }
                *reinterpret_cast<uint4*>(A + kmajor_off(row, c0 + c * 8)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        tc_fence_before();
        fence_async_smem();
        sync();
        // 4. h2 W3^T (16 padded outputs) into accumulator columns 0..15
        if (gt == 0) {
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < NH / 16; ++kk)
                tc_mma(tmem, sdesc(a_addr + kk * 2 * kLbo, kLbo, kSbo), sdesc(w3_addr + kk * 2 * kLbo, kLbo, kSbo),
                       idesc_bf16(128, 16), kk > 0 ? 1u : 0u);
            tc_commit(bar);
        }
        if (!bar_wait(bar, parity)) S.abort[group] = 1;
        parity ^= 1;
        tc_fence_after();
        sync();
        if (S.abort[group]) break;
        if (half == 0) {
            float o8[8];
            tmem_ld8(tmem + lane_base, o8);
            if (valid)
#pragma unroll
                for (int o = 0; o < NO; ++o) y[p * NO + o] = o8[o] + S.b3[o];
        }
        tc_fence_before();
        sync();
    }
    if (S.abort[group]) {
        // a wait expired: mark this block's remaining outputs and report
        if (gt == 0) atomicOr(err, 1);
        for (long long tile = first; tile < n_tiles; tile += stride) {
            const long long p = tile * kTcRows + row;
            if (half == 0 && p < n)
                for (int o = 0; o < NO; ++o) y[p * NO + o] = __int_as_float(0x7fc00000);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(S.tmem), "r"(128 * kTcGroups) : "memory");
    }
}

// ------------------------------------------------------------------ standardization
// The caller's affine standardizations folded into the parameters (one
// thread per parameter, float64 arithmetic rounded once): inputs x_std =
// (x - xm) / xs enter layer 1, outputs y = y_std ys + ym leave layer 3.
struct Affine {
    double xm[NI], xs[NI], ym[NO], ys[NO];
};
__global__ void k_fold(const float* __restrict__ th, Affine a, float* __restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= NP) return;
    double v = (double)th[k];
    if (k < OFF_B1) {
        v /= a.xs[k % NI];
    } else if (k < OFF_W2) {
        const int o = k - OFF_B1;
        for (int i = 0; i < NI; ++i) v -= (double)th[OFF_W1 + o * NI + i] * a.xm[i] / a.xs[i];
    } else if (k >= OFF_W3 && k < OFF_B3) {
        v *= a.ys[(k - OFF_W3) / NH];
    } else if (k >= OFF_B3) {
        const int o = k - OFF_B3;
        v = v * a.ys[o] + a.ym[o];
    }
    out[k] = (float)v;
}

// The network's inputs of transport-data queries: log10(E/N in Td) and the
// O2 fraction, in float32 (the network's input precision; a float64
// logarithm would run on this GPU's slow float64 units).
__global__ void k_features(const double* __restrict__ en, const double* __restrict__ f, float* __restrict__ x,
                           long long n, bool wide) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    auto one = [&](long long i) {
        reinterpret_cast<float2*>(x)[i] = make_float2(log10f((float)en[i]), (float)f[i]);
    };
    if (!wide) {
        for (long long i = t; i < n; i += step) one(i);
        return;
    }
    for (long long i = t; i < n / 4; i += step) {
        const double2* q = reinterpret_cast<const double2*>(en) + 2 * i;
        const double2* g = reinterpret_cast<const double2*>(f) + 2 * i;
        const double2 a = q[0], b = q[1], c = g[0], d = g[1];
        float4* o = reinterpret_cast<float4*>(x) + 2 * i;
        o[0] = make_float4(log10f((float)a.x), (float)c.x, log10f((float)a.y), (float)c.y);
        o[1] = make_float4(log10f((float)b.x), (float)d.x, log10f((float)b.y), (float)d.y);
    }
    if (t < (n & 3)) one((n & ~3ll) + t);
}

}  // namespace mlp

// ------------------------------------------------------------------ C ABI
using namespace mlp;

namespace {

size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

struct TrainWs {
    __nv_bfloat16* w2b;
    float *gw2, *head, *l1;  // partial sums
    int* err;
    int splits, n_head, n_l1;
};

// Layout of the workspace for n points (base null: sizes only).
size_t carve(void* base, int n, TrainWs* w) {
    uintptr_t p = (uintptr_t)base;
    const uintptr_t p0 = p;
    auto take = [&](size_t b) {
        void* r = (void*)p;
        p += al256(b);
        return r;
    };
    w->splits = n >= kSplitPts ? n / kSplitPts : 1;
    w->n_head = w->n_l1 = n / kPts;
    w->w2b = (__nv_bfloat16*)take(NH * NH * 2);
    w->gw2 = (float*)take((size_t)w->splits * NH * NH * 4);
    w->head = (float*)take((size_t)w->n_head * kHeadPart * 4);
    w->l1 = (float*)take((size_t)w->n_l1 * kL1Part * 4);
    w->err = (int*)take(64);
    return (size_t)(p - p0);
}

Parts parts_of(const TrainWs& w) {
    Parts P;
    P.gw2 = w.gw2;
    P.head = w.head;
    P.l1 = w.l1;
    P.splits = w.splits;
    P.n_head = w.n_head;
    P.n_l1 = w.n_l1;
    return P;
}

// Forward and backward over the batch: leaves the partial sums in the workspace.
cudaError_t backprop(const float* th, const float* x, const float* t, int n, const TrainWs& w, cudaStream_t s) {
    const float inv6n = 1.0f / (6.0f * (float)n);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n / kPts);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = sizeof(TrainSmem);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = n / kPts / w.splits;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_backprop, th, (const __nv_bfloat16*)w.w2b, x, t, inv6n, w.head, w.l1, w.gw2);
}
cudaError_t backprop_prepare(const float* params, const TrainWs& w, cudaStream_t s) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_backprop, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
    if (e == cudaSuccess) k_prep<<<(NH * NH + 255) / 256, 256, 0, s>>>(params, w.w2b);
    return e;
}

bool train_size_ok(int n) { return n >= 64 && n % 64 == 0 && (n < 256 || n % 256 == 0); }

}  // namespace

extern "C" size_t mlp_workspace_bytes(int n_max) {
    if (n_max < 0 || (n_max > 0 && !train_size_ok(n_max))) return 0;
    TrainWs w;
    return carve(nullptr, n_max > 0 ? n_max : 64, &w);
}

extern "C" int mlp_forward_variant(const float* params, const float* x, float* y, long long n, int variant,
                                   void* ws, size_t ws_bytes, pic_stream_t stream) {
    if (!params || !x || !y || n < 0 || !ws || ((uintptr_t)ws & 255) || ws_bytes < mlp_workspace_bytes(0) ||
        (variant != 0 && variant != 1))
        return PIC_ERR_ARG;
    if (n == 0) return PIC_OK;
    cudaStream_t s = (cudaStream_t)stream;
    TrainWs w;
    carve(ws, 64, &w);
    k_prep<<<(NH * NH + 255) / 256, 256, 0, s>>>(params, w.w2b);
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (variant == 0) {
        const int smem = (int)sizeof(TcSmem) + 1024;
        if (cudaFuncSetAttribute(k_infer_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
            return PIC_ERR_CUDA;
        // one block an SM (shared memory, 512 tensor-memory columns); few tiles are spread over the SMs
        const long long tiles = (n + kTcRows - 1) / kTcRows, blocks = tiles < sms ? tiles : sms;
        k_infer_tc<<<(unsigned)blocks, kTcThreads, smem, s>>>(params, w.w2b, x, y, n, w.err);
    } else {
        const int smem = (int)sizeof(InfSmem);
        if (cudaFuncSetAttribute(k_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
            return PIC_ERR_CUDA;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_infer, kInfWarps * 32, smem);
        const long long tiles = (n + 15) / 16;
        long long blocks = (long long)sms * (per_sm > 0 ? per_sm : 1);
        if (blocks * kInfWarps > tiles) blocks = (tiles + kInfWarps - 1) / kInfWarps;
        k_infer<<<(unsigned)blocks, kInfWarps * 32, smem, s>>>(params, w.w2b, x, y, n);
    }
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

extern "C" int mlp_fold_standardization(const float* params, const double x_mean[2], const double x_scale[2],
                                        const double y_mean[6], const double y_scale[6], float* out,
                                        pic_stream_t stream) {
    if (!params || !out || params == out || !x_mean || !x_scale || !y_mean || !y_scale) return PIC_ERR_ARG;
    mlp::Affine a;
    for (int i = 0; i < mlp::NI; ++i) {
        if (!(x_scale[i] != 0.0) || !isfinite(x_scale[i]) || !isfinite(x_mean[i])) return PIC_ERR_ARG;
        a.xm[i] = x_mean[i];
        a.xs[i] = x_scale[i];
    }
    for (int o = 0; o < mlp::NO; ++o) {
        if (!isfinite(y_scale[o]) || !isfinite(y_mean[o])) return PIC_ERR_ARG;
        a.ym[o] = y_mean[o];
        a.ys[o] = y_scale[o];
    }
    mlp::k_fold<<<(mlp::NP + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, a, out);
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

// Four points a thread from 16-byte aligned arrays: more bytes in flight (1.7e7 points 83 us with one, 59 now);
// below 2^18 points one a thread fills more SMs.
constexpr long long kWideFeatures = 1ll << 18;
extern "C" int mlp_features(const double* EN_Td, const double* f_o2, float* x, long long n, pic_stream_t stream) {
    if (n < 0 || (n > 0 && (!EN_Td || !f_o2 || !x))) return PIC_ERR_ARG;
    if (n == 0) return PIC_OK;
    const bool wide = (((uintptr_t)EN_Td | (uintptr_t)f_o2 | (uintptr_t)x) & 15) == 0 && n >= kWideFeatures;
    long long g = (wide ? n / 4 + 255 : n + 255) / 256;
    if (g > 65535) g = 65535;
    mlp::k_features<<<(unsigned)g, 256, 0, (cudaStream_t)stream>>>(EN_Td, f_o2, x, n, wide);
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

extern "C" int mlp_forward(const float* params, const float* x, float* y, long long n, void* ws, size_t ws_bytes,
                           pic_stream_t stream) {
    return mlp_forward_variant(params, x, y, n, 0, ws, ws_bytes, stream);
}

extern "C" int mlp_loss_grad(const float* params, const float* x, const float* t, int n, float* grad, float* loss,
                             void* ws, size_t ws_bytes, pic_stream_t stream) {
    if (!params || !x || !t || !grad || !ws || ((uintptr_t)ws & 255) || !train_size_ok(n) ||
        ws_bytes < mlp_workspace_bytes(n))
        return PIC_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    TrainWs w;
    carve(ws, n, &w);
    if (backprop_prepare(params, w, s) != cudaSuccess || backprop(params, x, t, n, w, s) != cudaSuccess)
        return PIC_ERR_CUDA;
    k_grad_out<<<kParamBlocks, kParamThreads, 0, s>>>(parts_of(w), grad, loss, 1.0f / (6.0f * (float)n));
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

extern "C" int mlp_train(float* params, float* m, float* v, int step0, const float* x, const float* t, int n,
                         int n_steps, float lr, float beta1, float beta2, float eps, float* loss, void* ws,
                         size_t ws_bytes, pic_stream_t stream) {
    if (!params || !m || !v || !x || !t || !ws || ((uintptr_t)ws & 255) || !train_size_ok(n) || n_steps < 0 ||
        step0 < 0 || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0) ||
        ws_bytes < mlp_workspace_bytes(n))
        return PIC_ERR_ARG;
    if (n_steps == 0) return PIC_OK;
    cudaStream_t s = (cudaStream_t)stream;
    TrainWs w;
    carve(ws, n, &w);
    const float inv6n = 1.0f / (6.0f * (float)n);
    // two launches a step, queued faster than they run (a recorded graph of them would cost more than it saves)
    cudaError_t e = backprop_prepare(params, w, s);
    for (int k = 0; k < n_steps && e == cudaSuccess; ++k) {
        e = backprop(params, x, t, n, w, s);
        if (e == cudaSuccess)
            e = pic::launch_pdl(k_adam, dim3(kParamBlocks), dim3(kParamThreads), 0, s, parts_of(w), params, m, v,
                                step0 + k + 1, lr, beta1, beta2, eps, w.w2b, loss, inv6n);
    }
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ERR_CUDA;
}

// Axisymmetric Poisson solve on an (r, z) mesh (see poisson_axi.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "graph_util.cuh"

namespace pic {

// Right-hand side of a solve: rho in C/m^3, or (rho null) the fixed-point
// charges of the grid, b = scale (q_pos - q_neg - q_e) with the ring volumes
// cancelled against the ring cells' factor.
struct AxiCharge {
    const double* rho;
    const long long *qe, *qp, *qn;
    double scale;
};

// Loop state of a device-driven axisymmetric solve (device memory).
struct AxiLoop {
    int cyc, trips, timeout, pad;
    int n_branch[2];
    double rel;
};

struct AxiMG : LaunchStatus {
    static constexpr int kMaxLevels = 14;
    int levels = 0;
    int lr[kMaxLevels], lz[kMaxLevels];
    double* e[kMaxLevels];
    double* g[kMaxLevels];
    uint8_t* m[kMaxLevels];
    double* rd[kMaxLevels];  // reciprocal diagonals by column: [nr] inside, [nr] at the z faces
    double *norms = nullptr, *r = nullptr, *p = nullptr, *q = nullptr, *w = nullptr;
    double* part = nullptr;   // per-block partial sums
    unsigned* ctr = nullptr;  // arrivals of their blocks
    int pre = 2, post = 2, coarse_sweeps = 64;
    long long launches = 0;
    bool persistent = false, masks_ready = false;
    AxiLoop* loop = nullptr;
    cudaStream_t cap_body[3] = {nullptr, nullptr, nullptr};
    // Streams for recording loop bodies (call before the caller's capture).
    int prepare_capture();
    void release();
    // Records the solve on the capturing stream cs: residual, an if node with
    // the first CG iteration, in it another with a device-side while loop over
    // the later ones (most coupled solves need one iteration), the gradient
    // and a report of cycles, relative residual, cycle-limit flag (err_bit
    // into *err_dst) and the kernels run in the nodes (added to
    // *kernels_dst).  No host synchronisation.  Returns PIC_OK or
    // PIC_ERR_CUDA / PIC_ERR_STATE (callers then use solve).
    int capture_solve(cudaStream_t cs, const AxiCharge& rho, double* phi, double h, double v_lo, double v_hi,
                      double v_mask, double rtol, int max_cycles, int packed_prec, void* E4, int* cycles_dst,
                      double* rel_dst, unsigned* err_dst, unsigned err_bit, unsigned long long* kernels_dst,
                      long long* fixed_kernels);

    void plan(int nr, int nz);
    // The coarsest level is solved by one block: at most 4096 cells.
    static bool supported(int nr, int nz);
    static size_t bytes(int nr, int nz);
    size_t carve(void* base, int nr, int nz);
    cudaError_t build_masks(const uint8_t* mask, cudaStream_t s);
    int tail_level() const;  // first level of the one-block kernel (levels: none)
    void vcycle(cudaStream_t s);
    void iteration(cudaStream_t s, double* phi, bool first);
    // rho: charge [nz][nr]; phi: initial guess and solution;
    // E4 (optional): packed [nz][nr][4] (E_r, 0, E_z, 0) in float (packed_prec
    // 32) or double (64); Er, Ez: optional float planes.  Returns PIC_OK,
    // PIC_ERR_TIMEOUT or PIC_ERR_CUDA.
    int solve(const AxiCharge& rho, const uint8_t* mask, double* phi, double h, double v_lo, double v_hi,
              double v_mask, double rtol, int max_cycles, int packed_prec, void* E4, float* Er, float* Ez,
              cudaStream_t s, int* cycles_out, double* rel_out, double* host_norms);
};

}  // namespace pic

// Krylov pressure solver (paper, Section 4: the model's second pressure
// solver, BiCGStab on the same Poisson problem as the FFT solver).  Host-side
// interface between the C ABI (monc_proj.cu) and the kernels (kern_krylov.cu).
#pragma once
#include <cstddef>
#include <vector>
#include <cuda_runtime.h>

namespace mp {

struct KrylovProblem {
    int nx, ny, nz;
    int nsm;                      // SMs of the device (grid of the streaming kernels)
    double dx, dy;
    // device tables of the plan
    const void* tables;           // krylov_tables, in the vectors' type
    const double* idzn;           // [nz+1] 1/dzn[k]
    // fields (FP32 when fp32, else FP64): u, v, phi [nz][ny][nx], w [nz+1][ny][nx]
    int fp32;
    const void* u; const void* v; const void* w;
    void* u_out; void* v_out; void* w_out; void* phi_out;           // phi_out may be null
    void* workspace;
    double tol;
    int max_iter;
    int precond;                  // 0: none, 1: vertical lines
};

struct KrylovResult {
    int iterations;
    double rel_residual;
    int status;                   // 0 converged, 1 iteration limit, 2 breakdown
};

// The vertical tables of a plan (host arrays as in the plan's blob).
std::vector<double> krylov_tables(int nz, double dx, double dy, const double* acoef, const double* svol,
                                  const double* rflo, const double* rfhi);

size_t krylov_workspace_bytes(int nx, int ny, int nz, int nsm, bool fp32);

// Runs the whole solve on `st`, reading the residual back every few
// iterations (the calling thread waits on the stream).  Returns a cudaError_t.
cudaError_t krylov_run(const KrylovProblem& kp, cudaStream_t st, KrylovResult* res);

}  // namespace mp

// solver_rowc.cu -- the row layout over a cluster of CTAs (solver_row.cuh, CLU):
// N = 2048 and 4096, intensity cost.
#include "solver_row.cuh"

namespace tmr {

int solver_rowc_masks(int N, int J) { return J >= 1 && J <= kMaxMasks ? rowc_masks(N, J) : 0; }

size_t solver_rowc_smem(int N, int J, int m)
{
    const int JB = solver_rowc_masks(N, J);
    if (!JB) return 0;
    const int JC = J / JB;
    // N = 4096, J = 4, m = 6: the pairs leave the fields no room in tensor memory
    if (!row_fields_fit(row_shape(N, JB, (N + JC - 1) / JC), m, 0)) return (size_t)1 << 30;
    return N == 2048 ? rowc_smem<2048>(J) : rowc_smem<4096>(J);
}

cudaError_t launch_solver_rowc(int N, const SolverParams &p, cudaStream_t s, int *clusters_out)
{
    if (!solver_rowc_masks(N, p.J)) return cudaErrorInvalidValue;
    return N == 2048 ? launch_solver_rowc_t<2048>(p, s, clusters_out) : launch_solver_rowc_t<4096>(p, s, clusters_out);
}

}  // namespace tmr

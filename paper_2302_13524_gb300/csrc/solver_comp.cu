// solver_comp.cu -- the cluster solver for composite lengths N = A B (XfComp), one
// mask per CTA, with the intensity cost.
#include "solver_impl.cuh"

namespace tmr {

template <int TEAMS>
static size_t smem_t(int N, int J, int m) { return solver_smem<XfComp<TEAMS>, 1>(N, J, m); }

size_t solver_comp_smem(int N, int J, int m)
{
    int A = 0, B = 0;
    if (!comp_shape(N, &A, &B)) return 0;
    switch (comp_teams(A)) {
    case 2: return smem_t<2>(N, J, m);
    case 4: return smem_t<4>(N, J, m);
    case 8: return smem_t<8>(N, J, m);
    case 12: return smem_t<12>(N, J, m);
    case 18: return smem_t<18>(N, J, m);
    case 24: return smem_t<24>(N, J, m);
    default: return smem_t<32>(N, J, m);
    }
}

cudaError_t launch_solver_comp(int N, const SolverParams &p, cudaStream_t s, int *clusters_out)
{
    int A = 0, B = 0;
    if (!comp_shape(N, &A, &B)) return cudaErrorInvalidValue;
    switch (comp_teams(A)) {
    case 2: return launch_solver_t<XfComp<2>, 1>(p, s, clusters_out);
    case 4: return launch_solver_t<XfComp<4>, 1>(p, s, clusters_out);
    case 8: return launch_solver_t<XfComp<8>, 1>(p, s, clusters_out);
    case 12: return launch_solver_t<XfComp<12>, 1>(p, s, clusters_out);
    case 18: return launch_solver_t<XfComp<18>, 1>(p, s, clusters_out);
    case 24: return launch_solver_t<XfComp<24>, 1>(p, s, clusters_out);
    default: return launch_solver_t<XfComp<32>, 1>(p, s, clusters_out);
    }
}

}  // namespace tmr

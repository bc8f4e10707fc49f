// solver_comp_amp.cu -- the cluster solver for composite lengths N = A B (XfComp), one
// mask per CTA, with the amplitude cost.
#include "solver_impl.cuh"

namespace tmr {

cudaError_t launch_solver_comp_amp(int N, const SolverParams &p, cudaStream_t s, int *clusters_out)
{
    int A = 0, B = 0;
    if (!comp_shape(N, &A, &B)) return cudaErrorInvalidValue;
    switch (comp_teams(A)) {
    case 2: return launch_solver_t<XfComp<2>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    case 4: return launch_solver_t<XfComp<4>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    case 8: return launch_solver_t<XfComp<8>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    case 12: return launch_solver_t<XfComp<12>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    case 18: return launch_solver_t<XfComp<18>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    case 24: return launch_solver_t<XfComp<24>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    default: return launch_solver_t<XfComp<32>, 1, COST_AMPLITUDE>(p, s, clusters_out);
    }
}

}  // namespace tmr

// solver_row_regs.cu -- the one-CTA-per-row solver (solver_row.cuh) with the row's
// fields kept in registers, both costs: for the shapes whose pairs leave them no
// room in tensor memory (N = 2048 with J = 3 and m >= 5, or J = 4 and m = 6), and
// those where their columns would cost a resident CTA (N = 512 and 1024 with
// J = 4 and m = 6; some with m <= 4).
#include "solver_row.cuh"

namespace tmr {

template <int COST>
static cudaError_t launch_regs(int N, const SolverParams &p, cudaStream_t s, int *ctas_out)
{
    switch (N) {
    case 512: return launch_solver_row_zt<512, COST, false>(p, s, ctas_out);
    case 1024: return launch_solver_row_zt<1024, COST, false>(p, s, ctas_out);
    case 2048: return launch_solver_row_zt<2048, COST, false>(p, s, ctas_out);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_solver_row_regs(int N, const SolverParams &p, cudaStream_t s, int *ctas_out)
{
    return p.cost == COST_AMPLITUDE ? launch_regs<COST_AMPLITUDE>(N, p, s, ctas_out)
                                    : launch_regs<COST_INTENSITY>(N, p, s, ctas_out);
}

}  // namespace tmr

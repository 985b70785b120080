#include "solve_kernel.cuh"

namespace mvgd {
namespace solver {

mvgd_status launch_mixed_amg(int Q, const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s) {
    return dispatch_q<true, true>(Q, tab, ctl, budget, kmax, s);
}
int rhs_group_mixed_amg(int Q, int tiles, int kmax) { return rhs_group<true, true>(Q, tiles, kmax); }

}  // namespace solver
}  // namespace mvgd

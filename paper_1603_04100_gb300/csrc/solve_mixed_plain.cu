#include "solve_kernel.cuh"

namespace mvgd {
namespace solver {

mvgd_status launch_mixed_plain(int Q, const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s) {
    return dispatch_q<true, false>(Q, tab, ctl, budget, kmax, s);
}
int rhs_group_mixed_plain(int Q, int tiles, int kmax) { return rhs_group<true, false>(Q, tiles, kmax); }

}  // namespace solver
}  // namespace mvgd

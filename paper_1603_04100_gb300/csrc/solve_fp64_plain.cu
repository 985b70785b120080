#include "solve_kernel.cuh"

namespace mvgd {
namespace solver {

mvgd_status launch_fp64_plain(int Q, const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s) {
    return dispatch_q<false, false>(Q, tab, ctl, budget, kmax, s);
}
int rhs_group_fp64_plain(int Q, int tiles, int kmax) { return rhs_group<false, false>(Q, tiles, kmax); }

}  // namespace solver
}  // namespace mvgd

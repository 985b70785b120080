#include "solve_kernel.cuh"

namespace mvgd {
namespace solver {

template mvgd_status launch_solve<false, 8, true>(const ReqTable&, Ctl, int, int, cudaStream_t);

}  // namespace solver
}  // namespace mvgd

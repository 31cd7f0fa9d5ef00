#include "solve_persistent.h"
namespace pisp {
template int launch_solve_dir<double, true>(bool, const SolveArgs<double>&, int32_t, int32_t, bool, int32_t, cudaStream_t);
}

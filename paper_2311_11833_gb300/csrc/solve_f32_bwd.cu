#include "solve_persistent.h"
namespace pisp {
template int launch_solve_dir<float, false>(bool, const SolveArgs<float>&, int32_t, int32_t, bool, int32_t, cudaStream_t);
}

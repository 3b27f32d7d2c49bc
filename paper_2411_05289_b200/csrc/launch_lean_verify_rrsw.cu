#include "launch_lean_verify.cuh"

namespace spechub {

int launch_lean_verify_rrsw(int format, int cs, const RowArgs &a, unsigned rows, cudaStream_t s) {
    return launch_lean_verify_method<kRRSw>(format, cs, a, rows, s);
}

}  // namespace spechub

#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<8, false>(const DiagMacArgs&, bool, cudaStream_t);
}

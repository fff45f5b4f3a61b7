#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<2, false>(const DiagMacArgs&, bool, cudaStream_t);
}

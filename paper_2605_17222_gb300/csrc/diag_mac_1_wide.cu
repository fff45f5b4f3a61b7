#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<1, false>(const DiagMacArgs&, bool, cudaStream_t);
}

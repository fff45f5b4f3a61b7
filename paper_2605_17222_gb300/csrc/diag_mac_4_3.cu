#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<4, 3>(const DiagMacArgs&, cudaStream_t);
}

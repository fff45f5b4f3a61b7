#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<8, 3>(const DiagMacArgs&, cudaStream_t);
}

#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<8, 2>(const DiagMacArgs&, cudaStream_t);
}

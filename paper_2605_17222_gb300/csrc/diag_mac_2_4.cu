#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<2, 4>(const DiagMacArgs&, cudaStream_t);
}

#include "diag_mac.cuh"

namespace ckks {
template bool launch_ws<1, 4>(const DiagMacArgs&, cudaStream_t);
}

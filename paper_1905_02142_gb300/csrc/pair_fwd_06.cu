// Forward pair kernel of basis class 6 (max(n_max, l_max) rounded up to even), both paths.
#include "pair_fwd.cuh"

template cudaError_t sg_pair_forward_class<float, 6>(const FwdArgs<float>&, cudaStream_t);
template cudaError_t sg_pair_forward_class<double, 6>(const FwdArgs<double>&, cudaStream_t);

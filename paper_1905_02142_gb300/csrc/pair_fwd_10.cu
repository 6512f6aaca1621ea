// Forward pair kernel of basis class 10 (max(n_max, l_max) rounded up to even), both paths.
#include "pair_fwd.cuh"

template cudaError_t sg_pair_forward_class<float, 10>(const FwdArgs<float>&, cudaStream_t);
template cudaError_t sg_pair_forward_class<double, 10>(const FwdArgs<double>&, cudaStream_t);

// cluster_gauss.cu -- the thread-block-cluster kernels for Gaussian couplings (see cluster_icm.cu).
#define ICM_PART 2
#include "cluster_icm.cu"

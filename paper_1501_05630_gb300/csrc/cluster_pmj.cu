// cluster_pmj.cu -- the thread-block-cluster kernels for +-J couplings (see cluster_icm.cu).
#define ICM_PART 1
#include "cluster_icm.cu"

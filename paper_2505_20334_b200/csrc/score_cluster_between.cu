// The cluster scoring kernels for sizes between the powers of two (see score_cluster.cu), in a module of
// their own: CUDA loads a module whole when one of its kernels is first wanted.
#define LAQ_SIZES_BETWEEN
#include "score_cluster.cu"

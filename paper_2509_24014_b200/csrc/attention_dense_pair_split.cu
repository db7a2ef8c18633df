// The CTA-pair dense kernel for grids whose last clusters own 256 query rows instead of 512.
#define SPARSED_SPLIT_CLUSTERS
#include "attention_dense_pair.cu"

// Tile kernels of the fp64 storage mode (see lb_tile_impl.cuh).
#define LBGB_PREC LB_PREC_FP64
#define LBGB_NAME fp64
#define LBGB_BATCH
#include "lb_tile_impl.cuh"

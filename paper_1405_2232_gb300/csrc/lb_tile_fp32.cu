// Tile kernels of the fp32 storage mode (see lb_tile_impl.cuh).
#define LBGB_PREC LB_PREC_FP32
#define LBGB_NAME fp32
#define LBGB_BATCH
#include "lb_tile_impl.cuh"

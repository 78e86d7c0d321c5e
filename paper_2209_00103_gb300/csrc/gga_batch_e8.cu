// Batched growth of 8-byte elements (gga_batch_grow.cuh).
#define GGA_BATCH_E 8
#include "gga_batch_grow.cuh"

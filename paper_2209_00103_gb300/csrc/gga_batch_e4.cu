// Batched growth of 4-byte elements (gga_batch_grow.cuh).
#define GGA_BATCH_E 4
#include "gga_batch_grow.cuh"

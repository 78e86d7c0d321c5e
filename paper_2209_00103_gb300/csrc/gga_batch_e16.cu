// Batched growth of 16-byte elements (gga_batch_grow.cuh).
#define GGA_BATCH_E 16
#include "gga_batch_grow.cuh"

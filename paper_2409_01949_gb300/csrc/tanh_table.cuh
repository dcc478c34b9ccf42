// The table of the fixed-point tanh (fixed.cuh), written by tanh_table.py when
// the library is built: fx::kTanhRows rows of three words.
#pragma once

#include "fixed.cuh"

static __device__ const int4 kTanhTable[3 * fx::kTanhRows] = {
#include "tanh_table.inc"
};

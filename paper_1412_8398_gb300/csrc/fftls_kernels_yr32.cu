// Register x2 pass in float.
#define FFTLS_Y_REG
#include "fftls_strided.cuh"

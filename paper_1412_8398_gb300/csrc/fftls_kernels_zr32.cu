// Register x3 / Fourier pass in float.
#define FFTLS_Z_REG
#include "fftls_strided.cuh"

#define EPFFT_REAL double
#include "inst_resident_impl.cuh"

#define EPFFT_REAL float
#include "inst_resident_impl.cuh"

// Device and host functions of the kernels' headers, callable one at a time.
#include "cgks_kernels.cuh"

using namespace cgks;

extern "C" long long unit_fr_nrow(int dir, int na, int nb) { return fr_nrow(dir, na, nb); }
extern "C" int unit_descriptor_bytes() { return (int)sizeof(Work); }

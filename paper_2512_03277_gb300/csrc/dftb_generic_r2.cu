// The cluster kernel (dftb_generic.cuh) with two product entries per thread per pass, a choice of the tuner.
#include "dftb_generic.cuh"

const void *dftb_generic_kernel_r2() { return (const void *)k_dftb_generic<2>; }

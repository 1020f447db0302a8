// k-grid kernel of the periodic cells (dftb_periodic.cuh): problems up to 256 wide, two blocks per SM.
#include "dftb_periodic.cuh"

const void *pbc_kg_small() { return (const void *)k_dftb_periodic_kg<PShared, 2>; }

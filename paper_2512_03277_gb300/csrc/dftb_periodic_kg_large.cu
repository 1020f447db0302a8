// k-grid kernel of the periodic cells (dftb_periodic.cuh): problems up to 512 wide, one block per SM.
#include "dftb_periodic.cuh"

const void *pbc_kg_large() { return (const void *)k_dftb_periodic_kg<PSharedK, 1>; }

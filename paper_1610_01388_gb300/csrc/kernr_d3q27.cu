// Resident-run kernels of the D3Q27 lattice.
#include "kernels.cuh"

BLBM_DEFINE_RESIDENT_LAUNCHERS(D3Q27)

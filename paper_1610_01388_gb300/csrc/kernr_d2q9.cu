// Resident-run kernels of the D2Q9 lattice.
#include "kernels.cuh"

BLBM_DEFINE_RESIDENT_LAUNCHERS(D2Q9)

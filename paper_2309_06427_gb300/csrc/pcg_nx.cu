// PCG kernel instantiations for nx = SSPCG_NX (compiled once per nx, see build.py).
#include "pcg_nx.cuh"

SSPCG_INSTANTIATE_PCG(SSPCG_NX)

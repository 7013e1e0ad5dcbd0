// Tensor-core PnP-Nystra kernels for windows of 256 tokens: the team kernel
// (nystra_team.cuh) for m <= 32, the wide kernel (nystra_wide.cuh) for m = 64.
#include "nystra_tc.cuh"
#include "nystra_team.cuh"
#include "nystra_wide.cuh"

NYSTRA_TC_DEFINE(n256, 64, 4, __nv_bfloat16, __half, false)

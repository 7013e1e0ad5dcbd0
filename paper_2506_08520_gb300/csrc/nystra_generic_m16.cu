// Generic PnP-Nystra kernel (nystra_generic.cuh) for up to 16 landmarks.
#include "nystra_generic.cuh"

NYSTRA_GENERIC_DEFINE(16)

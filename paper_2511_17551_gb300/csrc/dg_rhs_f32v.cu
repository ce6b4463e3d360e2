// Mixed form, right-hand-side kernels of the production flux pair with Sutherland's law (variable
// viscosity), 3D one-gas Navier-Stokes.
#define DG_REAL float
#define DG_PREFIX dg_f32v
#define DG_GENERIC_ONLY 1
#define DG_SUTH_ONLY 1
#include <string.h>
#include "dg_rhs_impl.cuh"

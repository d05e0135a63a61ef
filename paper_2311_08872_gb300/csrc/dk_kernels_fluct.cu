// The level kernels of the fluctuation state, in an image of their own: a context
// loads only the kind of state that it has.
#define DK_FLUCT_BUILD
#include "dk_kernels.cu"

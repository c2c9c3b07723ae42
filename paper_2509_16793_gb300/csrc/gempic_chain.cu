// The march instantiations of the denoised chain (gempic_set_denoiser), the same march source
// with its chain hooks compiled in, and the 128 x 128 one for simulations with a bunch, built as
// a translation unit of their own so that they compile beside gempic_kernels.cu.  Only the
// templates and the entry points below are taken from that file here; its other definitions are
// compiled there.
#define GEMPIC_CHAIN_TU
#include "gempic_kernels.cu"

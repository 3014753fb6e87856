// NLS split-step kernels, complex64.
#define SPDBA_T float
#define SPDBA_PAIRS 1   // long signals: two pencils per thread
#include "nls_kernels.inc"

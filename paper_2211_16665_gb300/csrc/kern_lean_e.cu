// The lean E kernels for rows that are no multiple of four (kern_lean.cu), compiled beside the others.
#define CSEM_LEAN_UNIT 2
#include "kern_lean.cu"
